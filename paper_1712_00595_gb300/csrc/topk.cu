// Top-k query (ranking by score descending, then id ascending).
//
// Radix select over order-preserving 64-bit keys of the scores: each pass
// histograms the next digit of the keys that still match the selected prefix
// and keeps the digit holding the k-th largest key, until the remaining bin is
// small enough to sort, or holds a single key value. The survivors (keys at or
// above the prefix) are collected in any order, or, when a single key value has
// too many holders, counted and compacted in id order so that the smallest ids
// stay. One CTA narrows them to about k by radix select on (key, id) and sorts
// those by (key descending, id ascending).
//
// Every kernel serves a table of independent jobs (one score vector and its
// scratch each): blockIdx.y is the job, so the top-k of many seeds costs one
// launch sequence.
#include <algorithm>
#include <climits>

#include "common.cuh"
#include "kernels.h"

namespace osp {

namespace {
constexpr int kDigitBits = 12;
constexpr int kBins = 1 << kDigitBits;

__device__ __forceinline__ unsigned long long order_key(double x) {
  unsigned long long b = (unsigned long long)__double_as_longlong(x);
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

// The order of keys as signed numbers: three 32-bit instructions a score.
__device__ __forceinline__ long long signed_key(long long bits) {
  return bits ^ ((bits >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ unsigned long long key_of(long long s) {
  return (unsigned long long)s ^ 0x8000000000000000ull;
}

// Signed keys of eight of the n scores: pairs p, p + stride, .. p + 3 stride (score
// 2 p is x[0]). Returns bit q for x[q] being one of the n. Whole pairs of an aligned
// vector load 16 bytes each, past the L2's set of lines to keep, and without a test
// of each index: a pass over 32 vectors of 2^21 scores 157 us with guarded 8-byte
// loads, 88 so.
__device__ __forceinline__ unsigned load_keys(const double* __restrict__ r, long long p, int stride,
                                              int n, long long (&x)[8]) {
  const bool whole = 2 * (p + 3ll * stride) + 1 < n && ((uintptr_t)r & 15) == 0;
  if (__all_sync(0xffffffffu, whole)) {
    longlong2 v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = __ldcs(reinterpret_cast<const longlong2*>(r) + p + q * stride);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      x[2 * q] = signed_key(v[q].x);
      x[2 * q + 1] = signed_key(v[q].y);
    }
    return 0xFFu;
  }
  unsigned have = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const long long i = 2 * (p + (long long)(q >> 1) * stride) + (q & 1);
    const bool in = i < n;
    have |= (unsigned)in << q;
    x[q] = in ? signed_key(__double_as_longlong(__ldg(r + i))) : 0ll;
  }
  return have;
}

__device__ __forceinline__ void bin_range(const TopkState* st, unsigned long long* lo,
                                          unsigned long long* hi) {
  const int bits = st->bits;
  if (bits == 0) {
    *lo = 0ull;
    *hi = ~0ull;
  } else {
    *lo = st->prefix << (64 - bits);
    *hi = bits >= 64 ? *lo : (*lo | ((1ull << (64 - bits)) - 1));
  }
}
}  // namespace

__global__ void k_topk_reset(TopkJobs J) {
  const TopkJob& jb = J.j[blockIdx.y];
  for (int i = threadIdx.x; i < kBins; i += blockDim.x) jb.hist[i] = 0;
  if (threadIdx.x == 0) {
    TopkState* st = jb.st;
    st->prefix = 0;
    st->bits = 0;
    st->k_rem = J.k;
    st->done = 0;
    st->count = 0;
    st->kmin = ~0ull;
    st->kmax = 0ull;
    st->arrived = 0;
    st->ties = 0;
  }
}

// Histogram of the next digit over the keys that match the prefix; also the
// smallest and largest such key, so that a prefix holding one key value (ties,
// typically of zero scores) ends the selection at once.
// The last CTA of the job then picks the digit d that holds the k_rem-th largest
// key (the largest d whose bins d.. hold at least k_rem keys) and extends the
// prefix; a launch of its own for that cost about 3 us a digit.
__global__ void __launch_bounds__(256) k_topk_hist(TopkJobs J, int width, int cand_max) {
  __shared__ unsigned sh[kBins];
  __shared__ long long s_w[8];
  __shared__ int s_d, s_last;
  __shared__ long long s_above;
  const TopkJob& jb = J.j[blockIdx.y];
  TopkState* st = jb.st;
  if (st->done) return;
  for (int i = threadIdx.x; i < kBins; i += blockDim.x) sh[i] = 0;
  __syncthreads();
  const double* __restrict__ r = jb.src;
  const int n = J.n;
  const int bits = st->bits;
  const unsigned long long prefix = st->prefix;
  const int shift = 64 - bits - width;
  const int stride = gridDim.x * blockDim.x;
  const long long pairs = ((long long)n + 1) >> 1;
  const unsigned mask = (1u << width) - 1u;
  unsigned long long lo, hi;
  bin_range(st, &lo, &hi);
  const long long slo = (long long)key_of((long long)lo), shi = (long long)key_of((long long)hi);
  // smallest and largest key from the second digit on (in the first they would tell
  // a vector of equal scores only)
  long long kmin = LLONG_MAX, kmax = LLONG_MIN;
  for (long long b = blockIdx.x * blockDim.x + (threadIdx.x & ~31); b < pairs; b += 4ll * stride) {
    long long x[8];
    const unsigned have = load_keys(r, b + (threadIdx.x & 31), stride, n, x);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      if (!((have >> q) & 1u) || (bits != 0 && (x[q] < slo || x[q] > shi))) continue;
      atomicAdd(&sh[(unsigned)(key_of(x[q]) >> shift) & mask], 1u);
      if (bits != 0) {
        kmin = x[q] < kmin ? x[q] : kmin;
        kmax = x[q] > kmax ? x[q] : kmax;
      }
    }
  }
  if (bits != 0) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const long long a = __shfl_xor_sync(0xffffffffu, kmin, o);
      const long long b = __shfl_xor_sync(0xffffffffu, kmax, o);
      kmin = a < kmin ? a : kmin;
      kmax = b > kmax ? b : kmax;
    }
    if ((threadIdx.x & 31) == 0 && kmin <= kmax) {
      atomicMin(&st->kmin, key_of(kmin));
      atomicMax(&st->kmax, key_of(kmax));
    }
  }
  __syncthreads();
  const int nb = 1 << width;
  for (int i = threadIdx.x; i < nb; i += blockDim.x)
    if (sh[i]) atomicAdd(&jb.hist[i], sh[i]);
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(&st->arrived, 1) == (int)gridDim.x - 1;
    __threadfence();
  }
  __syncthreads();
  if (!s_last) return;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  for (int i = t; i < nb; i += blockDim.x) {
    sh[i] = __ldcg(jb.hist + i);
    jb.hist[i] = 0;
  }
  if (t == 0) {
    s_d = -1;
    s_above = 0;
  }
  __syncthreads();
  const int k_rem = st->k_rem;
  // thread t owns the bins [b0, b1) counted from the top: bin nb-1-q for q in [b0, b1)
  const int per = (nb + (int)blockDim.x - 1) / (int)blockDim.x;
  const int b0 = min(nb, t * per), b1 = min(nb, b0 + per);
  long long mine = 0;
  for (int q = b0; q < b1; ++q) mine += sh[nb - 1 - q];
  long long inc = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) s_w[w] = inc;
  __syncthreads();
  long long above = inc - mine;  // keys in the bins above b0
  for (int q = 0; q < w; ++q) above += s_w[q];
  for (int q = b0; q < b1; ++q) {
    const int d = nb - 1 - q;
    if (above < k_rem && above + sh[d] >= k_rem) {
      s_d = d;
      s_above = above;
    }
    above += sh[d];
  }
  __syncthreads();
  if (t == 0) {
    int d = s_d;
    long long ab = s_above;
    if (d < 0) {  // fewer than k_rem keys match: keep everything
      d = 0;
      ab = 0;
      for (int i = 0; i < nb; ++i) ab += sh[i];
    }
    st->k_rem = k_rem - (int)ab;
    st->prefix = (prefix << width) | (unsigned long long)d;
    st->bits = bits + width;
    // one key value left under the prefix (the last pass saw a single value)
    const bool one = __ldcg(&st->kmin) == __ldcg(&st->kmax);
    const bool small = (int)sh[d] <= cand_max;
    if (small || bits + width >= 64 || one) {
      st->done = 1;
      st->ties = !small;
    }
    st->kmin = ~0ull;
    st->kmax = 0ull;
    st->arrived = 0;
  }
}

// Survivors (keys at or above the prefix) in any order: at most k - 1 above the
// bin and cand_max in it.
__global__ void __launch_bounds__(256) k_topk_collect(TopkJobs J, int cap) {
  const TopkJob& jb = J.j[blockIdx.y];
  TopkState* st = jb.st;
  if (st->ties) return;
  const double* __restrict__ r = jb.src;
  const int n = J.n;
  unsigned long long lo, hi;
  bin_range(st, &lo, &hi);
  const int lane = threadIdx.x & 31;
  const int stride = gridDim.x * blockDim.x;
  const long long pairs = ((long long)n + 1) >> 1;
  const long long slo = (long long)key_of((long long)lo);
  // whole warps stay in the loop: the append below is warp-wide
  for (long long b = blockIdx.x * blockDim.x + (threadIdx.x & ~31); b < pairs; b += 4ll * stride) {
    long long x[8];
    const unsigned have = load_keys(r, b + lane, stride, n, x);
    unsigned in = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) in |= (unsigned)(x[q] >= slo) << q;
    in &= have;
    if (!__any_sync(0xffffffffu, in)) continue;  // survivors are rare
    unsigned m[8];
    int tot = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      m[q] = __ballot_sync(0xffffffffu, (in >> q) & 1u);
      tot += __popc(m[q]);
    }
    int at = 0;
    if (lane == 0) at = atomicAdd(&st->count, tot);
    at = __shfl_sync(0xffffffffu, at, 0);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int p = at + __popc(m[q] & lanemask_lt());
      if ((in >> q) & 1u && p < cap) {
        jb.keys[p] = key_of(x[q]);
        jb.ids[p] = (int)(2 * (b + lane + (long long)(q >> 1) * stride) + (q & 1));
      }
      at += __popc(m[q]);
    }
  }
}

// Per chunk of kTopkChunk ids: how many keys lie above the selected bin and
// how many inside it. (A CTA takes many chunks: with one each, the CTAs of the
// jobs without ties took 27 us to start and leave, 32 jobs of 2^21 scores.)
__global__ void __launch_bounds__(1024) k_topk_count(TopkJobs J, int nb) {
  __shared__ int s_a, s_b;
  const TopkJob& jb = J.j[blockIdx.y];
  if (!jb.st->ties) return;
  const double* __restrict__ r = jb.src;
  const int n = J.n;
  unsigned long long lo, hi;
  bin_range(jb.st, &lo, &hi);
  for (int c = blockIdx.x; c < nb; c += gridDim.x) {
    if (threadIdx.x == 0) s_a = s_b = 0;
    __syncthreads();
    int a = 0, b = 0;
    const int base = c * kTopkChunk;
    for (int j = threadIdx.x; j < kTopkChunk; j += blockDim.x) {
      const int i = base + j;
      if (i >= n) break;
      const unsigned long long key = order_key(r[i]);
      a += key > hi;
      b += key >= lo && key <= hi;
    }
    a = warp_sum(a);
    b = warp_sum(b);
    if ((threadIdx.x & 31) == 0) {
      atomicAdd(&s_a, a);
      atomicAdd(&s_b, b);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      jb.blk_a[c] = s_a;
      jb.blk_b[c] = s_b;
    }
    __syncthreads();
  }
}

// One CTA per job (any multiple of 32 threads): exclusive scans of the chunk
// counts; how many bin keys to keep. Thread t scans a run of consecutive
// chunks, the runs' totals are scanned across the CTA.
__global__ void __launch_bounds__(1024) k_topk_scan(TopkJobs J, int nb, int cand_max) {
  __shared__ int s_a[32], s_b[32];
  const TopkJob& jb = J.j[blockIdx.y];
  if (!jb.st->ties) return;
  int* blk_above = jb.blk_a;
  int* blk_bin = jb.blk_b;
  const int nt = blockDim.x, t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int per = (nb + nt - 1) / nt;
  const int lo = min(nb, t * per), hi = min(nb, lo + per);
  int a = 0, b = 0;
  for (int i = lo; i < hi; ++i) {
    a += blk_above[i];
    b += blk_bin[i];
  }
  int ia = a, ib = b;  // inclusive scans over the warp, then over the warps
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int ya = __shfl_up_sync(0xffffffffu, ia, o), yb = __shfl_up_sync(0xffffffffu, ib, o);
    if (lane >= o) {
      ia += ya;
      ib += yb;
    }
  }
  if (lane == 31) {
    s_a[w] = ia;
    s_b[w] = ib;
  }
  __syncthreads();
  if (w == 0) {
    const int nw = nt >> 5;
    int xa = lane < nw ? s_a[lane] : 0, xb = lane < nw ? s_b[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int ya = __shfl_up_sync(0xffffffffu, xa, o), yb = __shfl_up_sync(0xffffffffu, xb, o);
      if (lane >= o) {
        xa += ya;
        xb += yb;
      }
    }
    s_a[lane] = xa;
    s_b[lane] = xb;
  }
  __syncthreads();
  int ra = (w ? s_a[w - 1] : 0) + ia - a, rb = (w ? s_b[w - 1] : 0) + ib - b;
  for (int i = lo; i < hi; ++i) {
    const int ta = blk_above[i], tb = blk_bin[i];
    blk_above[i] = ra;
    blk_bin[i] = rb;
    ra += ta;
    rb += tb;
  }
  if (t == nt - 1) {
    TopkState* st = jb.st;
    const int A = s_a[(nt >> 5) - 1], B = s_b[(nt >> 5) - 1];
    st->above = A;
    st->bin_count = B;
    // the whole bin when it is small; otherwise it is one key value and ties go by id
    st->keep = B <= cand_max ? B : min(B, st->k_rem);
    st->count = A + st->keep;
  }
}

// Ordered compaction: chunk by chunk in id order, keys above the bin go first,
// then the first `keep` keys of the bin.
__global__ void __launch_bounds__(1024) k_topk_emit(TopkJobs J, int nb) {
  __shared__ int s_w[2][32];
  __shared__ int s_run[2];
  const TopkJob& jb = J.j[blockIdx.y];
  const double* __restrict__ r = jb.src;
  const int n = J.n;
  const TopkState* st = jb.st;
  if (!st->ties) return;
  unsigned long long lo, hi;
  bin_range(st, &lo, &hi);
  const int above_total = st->above, keep = st->keep;
  unsigned long long* keys = jb.keys;
  int* ids = jb.ids;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int c = blockIdx.x; c < nb; c += gridDim.x) {
    int ra = jb.blk_a[c], rb = jb.blk_b[c];
    const int base = c * kTopkChunk;
    for (int round = 0; round < kTopkChunk / 1024; ++round) {
      const int i = base + round * 1024 + threadIdx.x;
      unsigned long long key = 0;
      int fa = 0, fb = 0;
      if (i < n) {
        key = order_key(r[i]);
        fa = key > hi;
        fb = key >= lo && key <= hi;
      }
      const unsigned ba = __ballot_sync(0xffffffffu, fa), bb = __ballot_sync(0xffffffffu, fb);
      if (lane == 0) {
        s_w[0][w] = __popc(ba);
        s_w[1][w] = __popc(bb);
      }
      __syncthreads();
      int pa = 0, pb = 0;
      for (int q = 0; q < w; ++q) {
        pa += s_w[0][q];
        pb += s_w[1][q];
      }
      pa += __popc(ba & lanemask_lt());
      pb += __popc(bb & lanemask_lt());
      if (fa) {
        keys[ra + pa] = key;
        ids[ra + pa] = i;
      }
      if (fb && rb + pb < keep) {
        keys[above_total + rb + pb] = key;
        ids[above_total + rb + pb] = i;
      }
      if (threadIdx.x == 0) {
        int ta = 0, tb = 0;
        for (int q = 0; q < 32; ++q) {
          ta += s_w[0][q];
          tb += s_w[1][q];
        }
        s_run[0] = ta;
        s_run[1] = tb;
      }
      __syncthreads();
      ra += s_run[0];
      rb += s_run[1];
      __syncthreads();
    }
  }
}

// One CTA per job: the survivors (up to cap) are narrowed to the k best, or to a
// set of at most 256 (or the next power of two above k) that holds them, by radix select on (key, then
// smaller id), eight bits a pass, with each thread's survivors in registers; a
// bitonic sort over the next power of two orders the rest, and the first k are
// written (to device or host-mapped memory). Sorting all survivors (up to k +
// 4,096) took 217 us for 32 jobs of k = 100.
constexpr int kTopkSortMin = 256;
__global__ void __launch_bounds__(1024) k_topk_sort(TopkJobs J, int cap) {
  extern __shared__ unsigned char smem[];
  __shared__ unsigned s_hist[256];
  __shared__ int s_pick, s_above, s_bin, s_n;
  const TopkJob& jb = J.j[blockIdx.y];
  const int cnt = min(jb.st->count, cap);  // count <= k + cand_max <= cap by construction
  constexpr int kPer = (kTopkMaxK + kTopkCand) / 1024;
  unsigned long long key[kPer];
  int id[kPer];
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const int i = threadIdx.x + 1024 * q;
    key[q] = i < cnt ? jb.keys[i] : 0ull;
    id[q] = i < cnt ? jb.ids[i] : 0x7FFFFFFF;
  }
  // digit p of (key, ~id), most significant first: 8 of the key, 4 of the id
  auto digit = [](unsigned long long k, int i, int p) -> unsigned {
    return p < 8 ? (unsigned)(k >> (56 - 8 * p)) & 255u : (~(unsigned)i >> (88 - 8 * p)) & 255u;
  };
  // an element's digits before p against those chosen: 1 above, 0 equal, -1 below
  unsigned long long ck = 0ull;  // chosen digits of the key ...
  unsigned ci = 0u;              // ... and of ~id
  auto place = [&](unsigned long long k, int i, int p) -> int {
    const unsigned long long a = p == 0 ? 0ull : p < 8 ? k >> (64 - 8 * p) : k;
    if (a != ck) return a > ck ? 1 : -1;
    if (p <= 8) return 0;
    const unsigned b = p == 12 ? ~(unsigned)i : ~(unsigned)i >> (96 - 8 * p);
    return b == ci ? 0 : b > ci ? 1 : -1;
  };
  int p = 0;
  int most = kTopkSortMin;  // enough to sort: the next power of two above k costs no more
  while (most < J.k) most <<= 1;
  int rem = J.k, left = cnt;  // rank to find among the elements that equal the chosen digits
  while (p < 12 && left > rem && J.k - rem + left > most) {
    for (int i = threadIdx.x; i < 256; i += blockDim.x) s_hist[i] = 0;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      if (1024 * q >= cnt) break;
      // survivors of one bin share their leading digits: one addition a warp then
      const bool in = threadIdx.x + 1024 * q < cnt && place(key[q], id[q], p) == 0;
      const unsigned dg = digit(key[q], id[q], p);
      const unsigned m = __ballot_sync(0xffffffffu, in);
      if (!m) continue;
      const unsigned d0 = __shfl_sync(0xffffffffu, dg, __ffs(m) - 1);
      if (__all_sync(0xffffffffu, !in || dg == d0)) {
        if ((threadIdx.x & 31) == 0) atomicAdd(&s_hist[d0], (unsigned)__popc(m));
      } else if (in) {
        atomicAdd(&s_hist[dg], 1u);
      }
    }
    __syncthreads();
    if (threadIdx.x < 32) {  // suffix sums from the largest digit; lane l owns digits 255 - 8 l ..
      unsigned c[8], sum = 0;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        c[q] = s_hist[255 - 8 * threadIdx.x - q];
        sum += c[q];
      }
      unsigned inc = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, inc, o);
        if ((int)threadIdx.x >= o) inc += y;
      }
      unsigned above = inc - sum;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if ((int)above < rem && (int)(above + c[q]) >= rem) {
          s_pick = 255 - 8 * threadIdx.x - q;
          s_above = (int)above;
          s_bin = (int)c[q];
        }
        above += c[q];
      }
    }
    __syncthreads();
    if (p < 8) ck = (ck << 8) | (unsigned)s_pick;
    else ci = (ci << 8) | (unsigned)s_pick;
    rem -= s_above;
    left = s_bin;
    ++p;
    __syncthreads();
  }
  // the kept ones: above the chosen digits or equal to them
  if (threadIdx.x == 0) s_n = 0;
  __syncthreads();
  const int kept = J.k < cnt ? J.k - rem + left : cnt;
  int N = 2;
  while (N < kept) N <<= 1;
  unsigned long long* sk = (unsigned long long*)smem;
  int* si = (int*)(sk + N);
#pragma unroll
  for (int q = 0; q < kPer; ++q)
    if (threadIdx.x + 1024 * q < cnt && place(key[q], id[q], p) >= 0) {
      const int at = atomicAdd(&s_n, 1);
      sk[at] = key[q];
      si[at] = id[q];
    }
  __syncthreads();
  for (int i = s_n + threadIdx.x; i < N; i += blockDim.x) {
    sk[i] = 0ull;
    si[i] = 0x7FFFFFFF;
  }
  __syncthreads();
  // "a before b": larger key, then smaller id
  for (int kk = 2; kk <= N; kk <<= 1) {
    for (int j = kk >> 1; j > 0; j >>= 1) {
      for (int t = threadIdx.x; t < (N >> 1); t += blockDim.x) {
        const int a = ((t & ~(j - 1)) << 1) | (t & (j - 1));
        const int b = a | j;
        const bool first = (a & kk) == 0;
        const bool b_before_a = sk[b] > sk[a] || (sk[b] == sk[a] && si[b] < si[a]);
        if (b_before_a == first) {
          const unsigned long long tk = sk[a];
          sk[a] = sk[b];
          sk[b] = tk;
          const int ti = si[a];
          si[a] = si[b];
          si[b] = ti;
        }
      }
      __syncthreads();
    }
  }
  const int kk = min(J.k, cnt);
  const double* norm = jb.norm;
  const double s = norm ? *norm : 1.0;
  for (int i = threadIdx.x; i < kk; i += blockDim.x) {
    const double v = jb.src[si[i]];
    jb.out_ids[i] = si[i];
    jb.out_sc[i] = norm ? (s > 0.0 ? v / s : 0.0) : v;
  }
  if (threadIdx.x == 0) *jb.out_k = kk;
}

// Seed-block columns in caller order: dst_j[int2ext[v]] = r[v Sp + col_j],
// walked in internal order, so that rows come in address order (the scattered
// writes land in L2). A warp takes 32 rows: lane = job reads one value of each
// (a row's sectors serve all jobs), a shared tile turns them, lane = row writes.
constexpr int kGatherWarps = 4;
__global__ void __launch_bounds__(32 * kGatherWarps) k_gather_cols(const double* __restrict__ r, int Sp,
                                                                   const int* __restrict__ int2ext,
                                                                   int n, int m, GatherJobs G) {
  __shared__ double tile[kGatherWarps][32][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int col = G.col[lane];  // zero above m
  double(*T)[33] = tile[w];
  for (int v0 = (blockIdx.x * kGatherWarps + w) * 32; v0 < n; v0 += gridDim.x * kGatherWarps * 32) {
    const int rows = min(32, n - v0);
    const double* p = r + (size_t)v0 * Sp + col;
    if (lane < m) {
#pragma unroll 8
      for (int q = 0; q < rows; ++q) T[lane][q] = p[(size_t)q * Sp];
    }
    __syncwarp();
    const int x = lane < rows ? int2ext[v0 + lane] : 0;
    if (lane < rows)
      for (int j = 0; j < m; ++j) G.dst[j][x] = T[j][lane];
    __syncwarp();
  }
}

// One column of the seed block in caller order, walked in internal order. kFar: the lines
// it touches do not stay in L2: four rows a thread in flight, past the L1, with a hint that
// keeps the L2 from fetching more of the row; else plain loads, whose 128-byte lines serve
// the next fifteen columns.
template <bool kFar>
__global__ void __launch_bounds__(256) k_gather_col(const double* __restrict__ r, int Sp, int col,
                                                    const int* __restrict__ int2ext, int n, double* out) {
  const int stride = gridDim.x * blockDim.x;
  constexpr int R = kFar ? 4 : 1;
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < n; b += R * stride) {
    double x[R];
    int to[R];
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const long long v = (long long)b + (long long)q * stride;
      to[q] = -1;
      if (v < n) {
        const double* p = r + (size_t)v * Sp + col;
        if constexpr (kFar)
          asm volatile("ld.global.nc.L1::no_allocate.L2::64B.f64 %0, [%1];" : "=d"(x[q]) : "l"(p));
        else
          x[q] = __ldg(p);
        to[q] = int2ext[v];
      }
    }
#pragma unroll
    for (int q = 0; q < R; ++q)
      if (to[q] >= 0) out[to[q]] = x[q];
  }
}

// Far when a column's 128-byte lines fill more than 60% of L2. Columns queried in turn,
// us each, far and near: 64 columns of 400,000 nodes 16.5 and 15.6, 700,000 19.5 and 22.4,
// 2^20 23 and 31, 2^21 36 and 57; near everywhere below, with the steps between: 100
// columns of 131,071 nodes there and back 5.6 and 5.3 ms, 256 of 2^18 from scratch 23.5 and
// 22.5.
void launch_gather_col(const double* r, int Sp, int col, const int* int2ext, int n, double* out,
                       int num_sms, int64_t l2_bytes, cudaStream_t st) {
  const bool far = (int64_t)n * 128 > l2_bytes * 6 / 10;
  (far ? k_gather_col<true> : k_gather_col<false>)<<<num_sms * 8, 256, 0, st>>>(r, Sp, col, int2ext, n, out);
}

int enqueue_topk_select(const TopkJobs& J, int num_sms, cudaStream_t st) {
  const int m = J.m;
  // about eight CTAs an SM over all jobs: every CTA clears and flushes a 16 KB histogram
  const int gx = max(1, min((J.n + 1023) / 1024, (num_sms * 8 + m - 1) / m));
  k_topk_reset<<<dim3(1, m), 1024, 0, st>>>(J);
  const int widths[6] = {12, 12, 12, 12, 12, 4};
  for (int w : widths) k_topk_hist<<<dim3(gx, m), 256, 0, st>>>(J, w, kTopkCand);
  k_topk_collect<<<dim3(gx, m), 256, 0, st>>>(J, kTopkMaxK + kTopkCand);
  const int nb = (J.n + kTopkChunk - 1) / kTopkChunk;
  const int gc = std::min(nb, std::max(1, num_sms * 2 / m));
  k_topk_count<<<dim3(gc, m), 1024, 0, st>>>(J, nb);
  k_topk_scan<<<dim3(1, m), 1024, 0, st>>>(J, nb, kTopkCand);
  k_topk_emit<<<dim3(gc, m), 1024, 0, st>>>(J, nb);
  return 11;
}

int enqueue_topk_sort(const TopkJobs& J, cudaStream_t st) {
  k_topk_sort<<<dim3(1, J.m), 1024, kTopkSortSmem, st>>>(J, kTopkMaxK + kTopkCand);
  return 1;
}

}  // namespace osp
