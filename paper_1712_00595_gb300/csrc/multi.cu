// Several seeds at once: the columns of an n x Sp block (Sp = 32 K) each hold
// the RWR vector of one seed, so every step of Algorithm 1 becomes a sparse
// matrix times a dense block (SpMM) and every gathered source brings K
// contiguous values per lane instead of one.
//
//   offset   q_offset = (1-c)(B~^T - A~^T) R_old over the changed rows u
//            (Sec. 3.1, 3.3): row u adds (1-c) R_old[u] / d'_u to every entry
//            of its new out-list and subtracts (1-c) R_old[u] / d_u from every
//            entry of its old out-list (old lists stay readable: the merge
//            writes new lists out of place); an entry in both lists gets the
//            difference in one addition. Targets get this call's stamp.
//   x(0)     one pass over all nodes: stamped rows move from xacc into R and
//            the first gather block y(0) = x(0) (1-c) / d; other rows of y(0)
//            are written as zero.
//   steps    pull only: x(i)[v] = sum over the in-list of v of y(i-1)[u],
//            a warp per node, lanes over columns; long in-lists in pieces.
//   stop     per column (Algorithm 1 loop test, do-while form): a column whose
//            ||x(i)||_1 <= eps stops adding and propagating; the call ends
//            when no column is left or at the iteration cap.
#include <cuda_bf16.h>

#include <type_traits>

#include "common.cuh"
#include "gridbar.cuh"
#include "kernels.h"

namespace osp {
namespace {

template <typename TY> struct AccOf { using type = float; };
template <> struct AccOf<double> { using type = double; };

__device__ __forceinline__ float to_acc(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float to_acc(float v) { return v; }
__device__ __forceinline__ double to_acc(double v) { return v; }
__device__ __forceinline__ __nv_bfloat16 from_acc(float v, __nv_bfloat16*) { return __float2bfloat16_rn(v); }
__device__ __forceinline__ float from_acc(float v, float*) { return v; }
__device__ __forceinline__ double from_acc(double v, double*) { return v; }

// K contiguous elements (K * sizeof(T) bytes, naturally aligned) through L2.
template <typename T, int K>
__device__ __forceinline__ void load_cg(const T* p, T (&out)[K]) {
  constexpr int B = K * (int)sizeof(T);
  if constexpr (B >= 16) {
#pragma unroll
    for (int i = 0; i < B / 16; ++i)
      reinterpret_cast<uint4*>(out)[i] = __ldcg(reinterpret_cast<const uint4*>(p) + i);
  } else if constexpr (B == 8) {
    *reinterpret_cast<uint2*>(out) = __ldcg(reinterpret_cast<const uint2*>(p));
  } else if constexpr (B == 4) {
    *reinterpret_cast<unsigned*>(out) = __ldcg(reinterpret_cast<const unsigned*>(p));
  } else {
    *reinterpret_cast<unsigned short*>(out) = __ldcg(reinterpret_cast<const unsigned short*>(p));
  }
}

template <typename T, int K>
__device__ __forceinline__ void store_k(T* p, const T (&v)[K]) {
  constexpr int B = K * (int)sizeof(T);
  if constexpr (B >= 16) {
#pragma unroll
    for (int i = 0; i < B / 16; ++i)
      reinterpret_cast<uint4*>(p)[i] = reinterpret_cast<const uint4*>(v)[i];
  } else if constexpr (B == 8) {
    *reinterpret_cast<uint2*>(p) = *reinterpret_cast<const uint2*>(v);
  } else if constexpr (B == 4) {
    *reinterpret_cast<unsigned*>(p) = *reinterpret_cast<const unsigned*>(v);
  } else {
    *reinterpret_cast<unsigned short*>(p) = *reinterpret_cast<const unsigned short*>(v);
  }
}

__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}

// ---------------------------------------------------------------------------
// L2 eviction priorities. Source rows of the gather block whose internal id is
// below PropParams::hot_n (with the degree node order: the most-read rows) are
// loaded with evict_last, so that they stay in L2 across a pull step; every
// other access of the step (cold source rows, score rows, residuals, the next
// gather block) touches its line once per step and is marked evict_first.
// All accesses go through L2 only (.cg): the gather blocks and score rows are
// rewritten inside the same persistent kernel.
// ---------------------------------------------------------------------------
struct L2Pol {
  unsigned long long keep;    // evict_last
  unsigned long long once;    // evict_first
  unsigned long long normal;  // evict_normal
};

// R += x without a return value, the line marked evict-first in L2: score rows
// are touched once per step and should not push gathered rows out of L2.
__device__ __forceinline__ void red_add_once(double* p, double x, unsigned long long pol) {
  asm volatile("red.global.add.L2::cache_hint.f64 [%0], %1, %2;" ::"l"(p), "d"(x), "l"(pol)
               : "memory");
}

__device__ __forceinline__ L2Pol make_l2pol() {
  L2Pol p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p.keep));
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p.once));
  asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p.normal));
  return p;
}

// K contiguous elements (K * sizeof(T) bytes, naturally aligned) through L2
// with an eviction policy.
template <typename T, int K>
__device__ __forceinline__ void ld_pol(const T* p, T (&out)[K], unsigned long long pol) {
  constexpr int B = K * (int)sizeof(T);
  static_assert(B == 2 || B == 4 || B == 8 || B % 16 == 0, "row slice size");
  if constexpr (B >= 16) {
#pragma unroll
    for (int i = 0; i < B / 16; ++i) {
      uint4 v;
      asm volatile("ld.global.cg.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
                   : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                   : "l"(reinterpret_cast<const uint4*>(p) + i), "l"(pol));
      reinterpret_cast<uint4*>(out)[i] = v;
    }
  } else if constexpr (B == 8) {
    uint2 v;
    asm volatile("ld.global.cg.L2::cache_hint.v2.u32 {%0, %1}, [%2], %3;"
                 : "=r"(v.x), "=r"(v.y)
                 : "l"(p), "l"(pol));
    *reinterpret_cast<uint2*>(out) = v;
  } else if constexpr (B == 4) {
    unsigned v;
    asm volatile("ld.global.cg.L2::cache_hint.u32 %0, [%1], %2;" : "=r"(v) : "l"(p), "l"(pol));
    *reinterpret_cast<unsigned*>(out) = v;
  } else {
    unsigned short v;
    asm volatile("ld.global.cg.L2::cache_hint.u16 %0, [%1], %2;" : "=h"(v) : "l"(p), "l"(pol));
    *reinterpret_cast<unsigned short*>(out) = v;
  }
}

template <typename T, int K>
__device__ __forceinline__ void st_pol(T* p, const T (&val)[K], unsigned long long pol) {
  constexpr int B = K * (int)sizeof(T);
  static_assert(B == 2 || B == 4 || B == 8 || B % 16 == 0, "row slice size");
  if constexpr (B >= 16) {
#pragma unroll
    for (int i = 0; i < B / 16; ++i) {
      const uint4 v = reinterpret_cast<const uint4*>(val)[i];
      asm volatile("st.global.L2::cache_hint.v4.u32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(
                       reinterpret_cast<uint4*>(p) + i),
                   "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "l"(pol)
                   : "memory");
    }
  } else if constexpr (B == 8) {
    const uint2 v = *reinterpret_cast<const uint2*>(val);
    asm volatile("st.global.L2::cache_hint.v2.u32 [%0], {%1, %2}, %3;" ::"l"(p), "r"(v.x), "r"(v.y),
                 "l"(pol)
                 : "memory");
  } else if constexpr (B == 4) {
    const unsigned v = *reinterpret_cast<const unsigned*>(val);
    asm volatile("st.global.L2::cache_hint.u32 [%0], %1, %2;" ::"l"(p), "r"(v), "l"(pol) : "memory");
  } else {
    const unsigned short v = *reinterpret_cast<const unsigned short*>(val);
    asm volatile("st.global.L2::cache_hint.u16 [%0], %1, %2;" ::"l"(p), "h"(v), "l"(pol) : "memory");
  }
}

template <typename T, int K>
__device__ __forceinline__ void zero_k(T (&out)[K]) {
  constexpr int B = K * (int)sizeof(T);
  if constexpr (B >= 16) {
#pragma unroll
    for (int i = 0; i < B / 16; ++i) reinterpret_cast<uint4*>(out)[i] = make_uint4(0, 0, 0, 0);
  } else if constexpr (B == 8) {
    *reinterpret_cast<uint2*>(out) = make_uint2(0, 0);
  } else if constexpr (B == 4) {
    *reinterpret_cast<unsigned*>(out) = 0u;
  } else {
    *reinterpret_cast<unsigned short*>(out) = 0;
  }
}

// bf16 gather rows carry the rounding residual of each stored value into the
// next step's rounding (error feedback, below); float and double rows do not.
template <typename TY> struct Feedback { static constexpr bool on = false; };
template <> struct Feedback<__nv_bfloat16> { static constexpr bool on = true; };

// Registers of one warp lane: KG columns of one column group.
template <typename TY, int KG>
struct ColGroup {
  static constexpr int G = 32 * KG;                      // columns of a group
  static constexpr int kRowBytes = G * (int)sizeof(TY);  // a group's slice of a gather row
  // rows gathered per batch of loads (more when a lane's share is small)
  static constexpr int kDepth = KG * (int)sizeof(TY) <= 8 ? 16 : 8;
};

// Sum of the gather rows of in-list entries p[0 .. len) into acc (this lane's
// KG columns; ys points at the lane's first column of row 0 of the group, rows
// Sp elements apart): 32 ids per coalesced load, then kDepth rows in flight.
template <typename TY, int KG, typename A>
__device__ __forceinline__ void sum_rows(const int* p, int len, const TY* ys, int Sp, A (&acc)[KG],
                                         int idx0, const L2Pol& pol, unsigned long long cold,
                                         int hot_n, bool on) {
  constexpr int D = ColGroup<TY, KG>::kDepth;
  const int lane = threadIdx.x & 31;
  for (int b = 0; b < len; b += 32) {
    const int cnt = min(32, len - b);
    // ids of the first block may come preloaded (idx0 >= 0 on every lane)
    const int idx = (b == 0 && __all_sync(0xffffffffu, idx0 >= 0)) ? idx0
                    : (lane < cnt ? __ldg(p + b + lane) : 0);
    int j = 0;
    for (; j + D <= cnt; j += D) {
      alignas(16) TY a[D][KG];
#pragma unroll
      for (int q = 0; q < D; ++q) {
        const int u = __shfl_sync(0xffffffffu, idx, j + q);
        if (on) ld_pol(ys + (size_t)u * Sp, a[q], u < hot_n ? pol.keep : cold);
        else zero_k(a[q]);
      }
#pragma unroll
      for (int k = 0; k < KG; ++k) {
        A t[D];
#pragma unroll
        for (int q = 0; q < D; ++q) t[q] = to_acc(a[q][k]);
#pragma unroll
        for (int h = D / 2; h > 0; h >>= 1)
#pragma unroll
          for (int q = 0; q < h; ++q) t[q] += t[q + h];
        acc[k] += t[0];
      }
    }
    for (; j + 4 <= cnt; j += 4) {
      alignas(16) TY a[4][KG];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int u = __shfl_sync(0xffffffffu, idx, j + q);
        if (on) ld_pol(ys + (size_t)u * Sp, a[q], u < hot_n ? pol.keep : cold);
        else zero_k(a[q]);
      }
#pragma unroll
      for (int k = 0; k < KG; ++k)
        acc[k] += (to_acc(a[0][k]) + to_acc(a[1][k])) + (to_acc(a[2][k]) + to_acc(a[3][k]));
    }
    for (; j < cnt; ++j) {
      const int u = __shfl_sync(0xffffffffu, idx, j);
      alignas(16) TY a[KG];
      if (on) ld_pol(ys + (size_t)u * Sp, a, u < hot_n ? pol.keep : cold);
      else zero_k(a);
#pragma unroll
      for (int k = 0; k < KG; ++k) acc[k] += to_acc(a[k]);
    }
  }
}

// x(i)[v] of this lane's KG columns of one group is acc. base / ybase: offset
// of the lane's first column in row v of R / of the group's gather block. rr: the row of R (loaded when the in-list is
// nonempty); eo: the carried residuals (bf16 rows). The running columns add x
// into R and |x| into l1; a node with out-edges (s != 0) writes its next
// gather row. With bf16 rows the value stored is the rounding of
// w = x s + e_old and the new residual is e = w - stored (error feedback:
// the stored values' rounding errors then telescope instead of adding up).
template <typename TY, int KG, typename A>
__device__ __forceinline__ void finish_slice(const Multi& M, size_t base, size_t ybase,
                                             const A (&acc)[KG], A s, bool has_in, double (&rr)[KG],
                                             const TY (&eo)[KG], unsigned act, TY* yd,
                                             double (&l1)[KG], const L2Pol& pol) {
  // a lane whose columns have all stopped moves nothing: its score entries
  // stay, and its gather entries are not read again in this call
  if (!act) return;
  if (has_in) {
#pragma unroll
    for (int k = 0; k < KG; ++k)
      if (act & (1u << k)) {
        const double x = (double)acc[k];
        rr[k] += x;
        l1[k] += fabs(x);
      }
    st_pol(M.r + base, rr, pol.once);
  }
  if (s != (A)0) {
    alignas(16) TY yv[KG];
    if constexpr (Feedback<TY>::on) {
      alignas(16) TY ev[KG];
#pragma unroll
      for (int k = 0; k < KG; ++k) {
        const float w = (float)(acc[k] * s) + __bfloat162float(eo[k]);
        yv[k] = __float2bfloat16_rn(w);
        ev[k] = __float2bfloat16_rn(w - __bfloat162float(yv[k]));
      }
      st_pol(reinterpret_cast<TY*>(M.e) + ybase, ev, pol.once);
    } else {
#pragma unroll
      for (int k = 0; k < KG; ++k) yv[k] = from_acc((A)(acc[k] * s), (TY*)nullptr);
    }
    st_pol(yd + ybase, yv, pol.once);
  }
}

template <typename A>
__device__ __forceinline__ A scale_of(const Dev& d, int v) {
  return std::is_same<A, double>::value ? (A)__ldg(d.scale_d + v) : (A)__ldg(d.scale_f + v);
}

// ---------------------------------------------------------------------------
// Team gather for bf16 rows of a 32-column group (64 bytes). The warp works as
// 4 teams of 8 lanes; lane (team t, sub s) loads columns [4 s, 4 s + 4) of a
// row (8 bytes), so one load instruction brings 4 rows. A window is 32
// consecutive positions of an edge stream (the in-lists of a run of nodes, or
// one piece of a long in-list); team t takes positions 8 t .. 8 t + 7 of it.
// Ids are loaded two windows ahead and rows one window ahead, so that up to
// 64 rows per warp are in flight whatever the list lengths.
// ---------------------------------------------------------------------------
struct TeamWin {
  uint2 v[8];  // this lane's 4 columns of its team's 8 rows (bf16 pairs)
};

__device__ __forceinline__ void team_load(TeamWin& w, int idx, const __nv_bfloat16* ysg, bool on,
                                          const L2Pol& pol, unsigned long long cold, int hot_n) {
  const int lane = threadIdx.x & 31;
  const int base = lane & 24, sub = lane & 7;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int u = __shfl_sync(0xffffffffu, idx, base + k);
    w.v[k] = make_uint2(0u, 0u);
    if (on && u >= 0) {
      const unsigned long long pp = u < hot_n ? pol.keep : cold;
      asm volatile("ld.global.cg.L2::cache_hint.v2.u32 {%0, %1}, [%2], %3;"
                   : "=r"(w.v[k].x), "=r"(w.v[k].y)
                   : "l"(ysg + (size_t)u * 32 + 4 * sub), "l"(pp));
    }
  }
}

// acc (4 columns) += one row slice of 4 bf16 values (the low half of each
// 32-bit word is the lower column); two packed f32x2 additions.
__device__ __forceinline__ void team_add(float (&acc)[4], uint2 x) {
  unsigned long long a01, a23, v01, v23;
  asm("mov.b64 %0, {%1, %2};" : "=l"(a01) : "f"(acc[0]), "f"(acc[1]));
  asm("mov.b64 %0, {%1, %2};" : "=l"(a23) : "f"(acc[2]), "f"(acc[3]));
  asm("mov.b64 %0, {%1, %2};" : "=l"(v01) : "r"(x.x << 16), "r"(x.x & 0xFFFF0000u));
  asm("mov.b64 %0, {%1, %2};" : "=l"(v23) : "r"(x.y << 16), "r"(x.y & 0xFFFF0000u));
  asm("add.rn.f32x2 %0, %0, %1;" : "+l"(a01) : "l"(v01));
  asm("add.rn.f32x2 %0, %0, %1;" : "+l"(a23) : "l"(v23));
  asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[0]), "=f"(acc[1]) : "l"(a01));
  asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[2]), "=f"(acc[3]) : "l"(a23));
}

// Sum of the rows of one piece of a long in-list (ids p[0 .. L)). Returns, in
// the lanes of team 0 (sub s: columns [4 s, 4 s + 4)), the sums over the
// whole piece; other lanes hold partial sums.
__device__ __forceinline__ void team_piece(const int* p, int L, const __nv_bfloat16* ysg, bool on,
                                           const L2Pol& pol, unsigned long long cold, int hot_n,
                                           float (&acc)[4]) {
  const int lane = threadIdx.x & 31;
  const int nwin = (L + 31) >> 5;
  auto id_of = [&](int i) -> int {
    const int q = i * 32 + lane;
    return (i < nwin && q < L) ? __ldg(p + q) : -1;
  };
#pragma unroll
  for (int c = 0; c < 4; ++c) acc[c] = 0.f;
  // ids run four windows ahead of the rows they name, rows one window ahead
  // of the additions
  int i0 = id_of(0), i1 = id_of(1), i2 = id_of(2), i3 = id_of(3);
  TeamWin A, B;
  team_load(A, i0, ysg, on, pol, cold, hot_n);
  for (int i = 0; i < nwin; i += 2) {
    const int i4 = id_of(i + 4);
    if (i + 1 < nwin) team_load(B, i1, ysg, on, pol, cold, hot_n);
#pragma unroll
    for (int k = 0; k < 8; ++k) team_add(acc, A.v[k]);
    if (i + 1 >= nwin) break;
    const int i5 = id_of(i + 5);
    if (i + 2 < nwin) team_load(A, i2, ysg, on, pol, cold, hot_n);
#pragma unroll
    for (int k = 0; k < 8; ++k) team_add(acc, B.v[k]);
    i1 = i3;
    i2 = i4;
    i3 = i5;
  }
  // the 4 teams' partial sums, combined in a fixed order
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], 8);
    acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], 16);
  }
}

// The in-lists of a run of up to 32 nodes as one edge stream: lane j holds
// node j's list length ll (0 to leave it out) and pool offset off; the sums
// per node and column land in acc_s[j * 32 + column] (shared memory of this
// warp, zeroed by the caller) through shared-memory atomics, one per column
// and run of a node's rows inside a team.
__device__ __forceinline__ void team_stream(const int* pool, int ll, unsigned off,
                                            const __nv_bfloat16* ysg, bool on, const L2Pol& pol,
                                            unsigned long long cold, int hot_n, float* acc_s) {
  const int lane = threadIdx.x & 31;
  const int base = lane & 24, sub = lane & 7;
  int incl = ll;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  const int P = incl - ll;
  const int E = __shfl_sync(0xffffffffu, incl, 31);
  if (E == 0) return;
  const int nwin = (E + 31) >> 5;
  // position q of the stream: node j = the last lane with P_j <= q, id from its list
  auto at = [&](int i, int& node) -> int {
    const int q = i * 32 + lane;
    int j = 0;
#pragma unroll
    for (int b = 16; b >= 1; b >>= 1) {
      const int Pc = __shfl_sync(0xffffffffu, P, j + b);
      if (Pc <= q) j += b;
    }
    const int Pj = __shfl_sync(0xffffffffu, P, j);
    const unsigned oj = __shfl_sync(0xffffffffu, off, j);
    node = -1;
    if (i >= nwin || q >= E) return -1;
    node = j;
    return __ldg(pool + oj + (unsigned)(q - Pj));
  };
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  int cur = -1;
  // edge: the current node has rows at the first or last row of one of this
  // team's runs, so other teams or windows may hold rows of it too (its sum
  // goes in by atomic additions); a node met only inside one run belongs to
  // this team alone and its sum is stored once
  bool edge = false;
  auto flush = [&]() {
    if (cur >= 0 && on) {
      float* a = acc_s + cur * 32 + 4 * sub;
      if (edge) {
#pragma unroll
        for (int c = 0; c < 4; ++c) atomicAdd(a + c, acc[c]);
      } else {
        *reinterpret_cast<float4*>(a) = make_float4(acc[0], acc[1], acc[2], acc[3]);
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[c] = 0.f;
  };
  auto eat = [&](const TeamWin& w, int nodes) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int jj = __shfl_sync(0xffffffffu, nodes, base + k);
      if (jj != cur) {
        flush();
        cur = jj;
        edge = k == 0;
      }
      team_add(acc, w.v[k]);
    }
    edge = true;  // the run's last node may go on in the next team or window
  };
  // ids (and nodes) run four windows ahead of the rows they name, rows one
  // window ahead of the additions
  int n0, n1, n2, n3, n4, n5;
  int i0 = at(0, n0), i1 = at(1, n1), i2 = at(2, n2), i3 = at(3, n3);
  TeamWin A, B;
  team_load(A, i0, ysg, on, pol, cold, hot_n);
  for (int i = 0; i < nwin; i += 2) {
    const int i4 = at(i + 4, n4);
    if (i + 1 < nwin) team_load(B, i1, ysg, on, pol, cold, hot_n);
    eat(A, n0);
    if (i + 1 >= nwin) break;
    const int i5 = at(i + 5, n5);
    if (i + 2 < nwin) team_load(A, i2, ysg, on, pol, cold, hot_n);
    eat(B, n1);
    n0 = n2;
    n1 = n3;
    n2 = n4;
    n3 = n5;
    i1 = i3;
    i2 = i4;
    i3 = i5;
  }
  flush();
}

// ---------------------------------------------------------------------------
// Narrow steps (bf16 rows, packed groups): once the only running columns are
// group slots 0..W-1 (W = 4 or 8), a step gathers W-value rows (8 or 16
// bytes) from a compact [node][W] block, whose rows of the nodes with
// out-edges (ids first in the degree order) mostly stay in L2, instead of the
// 64-byte slices of the 32-column group. Lane = position of the in-list
// stream of 32 nodes: each lane loads one row, a segmented warp scan per
// column sums each node's run, and the run's last lane adds it to the node's
// sums in shared memory; then lane = node finishes. A step reads the rows the
// step before it wrote, in that step's layout (the group layout, or a compact
// block of 8 or 4 columns: W only shrinks within a call).
// ---------------------------------------------------------------------------
template <int W>
struct Narrow {
  const __nv_bfloat16* src;  // gather rows of the previous step (row u at src + u stride)
  int stride;                // its row length: 32 (group 0 of the group layout), 8 or 4
  __nv_bfloat16* dst;        // next compact rows ([node][W])
  __nv_bfloat16* e;          // residual rows (group 0 of the group layout, slots 0..W-1 used)
  int col[W];                // columns of R held by slots 0..W-1
  unsigned act;              // bit c: column col[c] runs
};

__device__ __forceinline__ void bf16x4(uint2 x, float* f) {
  f[0] = __uint_as_float(x.x << 16);
  f[1] = __uint_as_float(x.x & 0xFFFF0000u);
  f[2] = __uint_as_float(x.y << 16);
  f[3] = __uint_as_float(x.y & 0xFFFF0000u);
}

template <int W>
struct NRow;
template <>
struct NRow<4> {
  uint2 v;
  __device__ __forceinline__ void load(const __nv_bfloat16* p) {
    v = __ldcg(reinterpret_cast<const uint2*>(p));
  }
  __device__ __forceinline__ void zero() { v = make_uint2(0u, 0u); }
  __device__ __forceinline__ void unpack(float (&f)[4]) const { bf16x4(v, f); }
};
template <>
struct NRow<8> {
  uint4 v;
  __device__ __forceinline__ void load(const __nv_bfloat16* p) {
    v = __ldcg(reinterpret_cast<const uint4*>(p));
  }
  __device__ __forceinline__ void zero() { v = make_uint4(0u, 0u, 0u, 0u); }
  __device__ __forceinline__ void unpack(float (&f)[8]) const {
    bf16x4(make_uint2(v.x, v.y), f);
    bf16x4(make_uint2(v.z, v.w), f + 4);
  }
};

__device__ __forceinline__ unsigned pack_bf16x2(float a, float b) {
  return (unsigned)__bfloat16_as_ushort(__float2bfloat16_rn(a)) |
         ((unsigned)__bfloat16_as_ushort(__float2bfloat16_rn(b)) << 16);
}

// Node v's sums x: R += x (running columns), |x| into l1, next compact row and
// residual w = x s + e_old (when v has out-edges).
template <int W>
__device__ __forceinline__ void narrow_finish(const Narrow<W>& N, const Multi& M, int v,
                                              const float (&x)[W], float s, bool has_in,
                                              double (&l1)[W]) {
  if (has_in) {
#pragma unroll
    for (int c = 0; c < W; ++c)
      if ((N.act >> c) & 1u) {
        atomicAdd(M.r + (size_t)v * M.Sp + N.col[c], (double)x[c]);
        l1[c] += fabs((double)x[c]);
      }
  }
  if (s != 0.f) {
    __nv_bfloat16* ep = N.e + (size_t)v * 32;
    NRow<W> eo;
    eo.load(ep);
    float e[W], y[W], r[W];
    eo.unpack(e);
#pragma unroll
    for (int c = 0; c < W; ++c) {
      const float w = x[c] * s + e[c];
      y[c] = __bfloat162float(__float2bfloat16_rn(w));
      r[c] = w - y[c];
    }
    if constexpr (W == 4) {
      *reinterpret_cast<uint2*>(N.dst + (size_t)v * 4) =
          make_uint2(pack_bf16x2(y[0], y[1]), pack_bf16x2(y[2], y[3]));
      *reinterpret_cast<uint2*>(ep) = make_uint2(pack_bf16x2(r[0], r[1]), pack_bf16x2(r[2], r[3]));
    } else {
      *reinterpret_cast<uint4*>(N.dst + (size_t)v * 8) =
          make_uint4(pack_bf16x2(y[0], y[1]), pack_bf16x2(y[2], y[3]), pack_bf16x2(y[4], y[5]),
                     pack_bf16x2(y[6], y[7]));
      *reinterpret_cast<uint4*>(ep) =
          make_uint4(pack_bf16x2(r[0], r[1]), pack_bf16x2(r[2], r[3]), pack_bf16x2(r[4], r[5]),
                     pack_bf16x2(r[6], r[7]));
    }
  }
}

// The in-lists of the nodes [vb, vb + 32) (lane j: list length ll, 0 for
// lists summed in pieces, at pool offset off) into acc_s[j * W + column]
// (this warp's shared memory, zeroed by the caller).
template <int W>
__device__ __forceinline__ void narrow_stream(const Narrow<W>& N, const int* pool, int ll,
                                              unsigned off, float* acc_s) {
  const int lane = threadIdx.x & 31;
  int incl = ll;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  const int P = incl - ll;
  const int E = __shfl_sync(0xffffffffu, incl, 31);
  // windows of 32 positions with their loads in flight together (narrower
  // rows leave registers for more)
  constexpr int R = W == 4 ? 8 : 6;
  for (int w0 = 0; w0 < E; w0 += 32 * R) {
    int node[R];
    NRow<W> row[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int q = w0 + 32 * r + lane;
      int j = 0;
#pragma unroll
      for (int b = 16; b >= 1; b >>= 1) {
        const int Pc = __shfl_sync(0xffffffffu, P, j + b);
        if (Pc <= q) j += b;
      }
      const int Pj = __shfl_sync(0xffffffffu, P, j);
      const unsigned oj = __shfl_sync(0xffffffffu, off, j);
      node[r] = q < E ? j : -1;
      row[r].zero();
      if (q < E) row[r].load(N.src + (size_t)__ldg(pool + oj + (unsigned)(q - Pj)) * N.stride);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (w0 + 32 * r >= E) break;  // warp-uniform
      float v[W];
      row[r].unpack(v);
      const int j = node[r];
      const int prev = __shfl_up_sync(0xffffffffu, j, 1);
      const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || prev != j);
      const int seg0 = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));
#pragma unroll
      for (int q = 1; q < 32; q <<= 1) {
#pragma unroll
        for (int c = 0; c < W; ++c) {
          const float t = __shfl_up_sync(0xffffffffu, v[c], q);
          if (lane - q >= seg0) v[c] += t;
        }
      }
      const int nxt = __shfl_down_sync(0xffffffffu, j, 1);
      if (j >= 0 && (lane == 31 || nxt != j)) {  // one run end per node and window
#pragma unroll
        for (int c = 0; c < W; ++c) acc_s[j * W + c] += v[c];
      }
      __syncwarp();
    }
  }
}

// One narrow step over the work items (long-list pieces, then tasks).
template <int W>
__device__ __forceinline__ void narrow_step(const Dev& d, const Multi& M, Narrow<W>& N, int n_items,
                                            int n_pieces, int hub_thr, int hub_piece, float* hub_acc,
                                            float* acc_s, double* my_part, Ctl* ctl) {
  const int lane = threadIdx.x & 31;
  const int Sp = M.Sp;
  double l1n[W];
#pragma unroll
  for (int c = 0; c < W; ++c) l1n[c] = 0.0;
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  for (int k = 0;; ++k) {
    int t = gw;  // the first item is the warp's own number, later ones come from the counter
    if (k > 0) {
      if (n_items <= nw) break;
      if (lane == 0) t = nw + atomicAdd(&ctl->ctr[1], 1);
      t = __shfl_sync(0xffffffffu, t, 0);
    }
    if (t >= n_items) break;
    if (t < n_pieces) {
      // a piece of a long in-list; the piece that completes the list finishes it
      const int h = __ldg(d.piece_hub + t);
      const int v = __ldg(d.hubs + h);
      const int piece = t - __ldg(d.hub_pstart + h);
      const int full = __ldg(d.len_c + v);
      const int* pl = d.pool_c + __ldg(d.off_c + v) + (unsigned)(piece * hub_piece);
      const int Lp = min(hub_piece, full - piece * hub_piece);
      float a[W];
#pragma unroll
      for (int c = 0; c < W; ++c) a[c] = 0.f;
      for (int b = 0; b < Lp; b += 128) {
        NRow<W> rw[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int e = b + 32 * r + lane;
          rw[r].zero();
          if (e < Lp) rw[r].load(N.src + (size_t)__ldg(pl + e) * N.stride);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          float f[W];
          rw[r].unpack(f);
#pragma unroll
          for (int c = 0; c < W; ++c) a[c] += f[c];
        }
      }
#pragma unroll
      for (int c = 0; c < W; ++c) a[c] = warp_sum(a[c]);
      float* ha = hub_acc + (size_t)h * Sp;  // group slots 0..W-1
      if (lane == 0) {
#pragma unroll
        for (int c = 0; c < W; ++c)
          if ((N.act >> c) & 1u) atomicAdd(ha + c, a[c]);
        __threadfence();
        const int np = (full + hub_piece - 1) / hub_piece;
        if (atomicAdd(&M.hub_cnt[h * 8], 1) == np - 1) {
          __threadfence();
          float x[W];
#pragma unroll
          for (int c = 0; c < W; ++c) {
            x[c] = __ldcg(ha + c);
            ha[c] = 0.f;
          }
          M.hub_cnt[h * 8] = 0;
          narrow_finish<W>(N, M, v, x, scale_of<float>(d, v), true, l1n);
        }
      }
      __syncwarp();
      continue;
    }
    const int task = t - n_pieces;
    const int c0t = __ldg(d.task_first + task), c1t = __ldg(d.task_first + task + 1);
    for (int vb = c0t; vb < c1t; vb += 32) {
      const int vl = vb + lane;
      int len = 0;
      unsigned off = 0;
      float sc = 0.f;
      if (vl < c1t) {
        len = __ldg(d.len_c + vl);
        off = __ldg(d.off_c + vl);
        sc = scale_of<float>(d, vl);
      }
      const bool mine = vl < c1t && len <= hub_thr;  // hubs go by pieces
      const bool fin = mine && (len > 0 || sc != 0.f);
      if (!__ballot_sync(0xffffffffu, fin)) continue;
#pragma unroll
      for (int c = 0; c < W; c += 4)
        reinterpret_cast<float4*>(acc_s)[(lane * W + c) / 4] = make_float4(0.f, 0.f, 0.f, 0.f);
      __syncwarp();
      narrow_stream<W>(N, d.pool_c, mine ? len : 0, off, acc_s);
      __syncwarp();
      if (fin) {
        float x[W];
#pragma unroll
        for (int c = 0; c < W; ++c) x[c] = acc_s[lane * W + c];
        narrow_finish<W>(N, M, vl, x, sc, len > 0, l1n);
      }
      __syncwarp();
    }
  }
#pragma unroll
  for (int c = 0; c < W; ++c) {
    const double sum = warp_sum(l1n[c]);
    if (lane == 0 && ((N.act >> c) & 1u)) atomicAdd(my_part + N.col[c], sum);
  }
}

// 16-byte asynchronous copy global -> shared (L2 only), and the wait for this
// thread's copies.
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(smem)), "l"(gmem)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// Whole last CTA: per-column sums of the partials (fixed order over CTAs),
// per-column stopping, the call's stop, the column groups still running and
// the history entry (max over the columns that ran the step). A column whose
// x(0) is exactly zero has only zero terms: under the eps rule its one
// do-while step is counted and it stops at once.
// s_sum (kPropThreads doubles) and s_key (kMaxSeeds doubles) are shared-memory
// scratch of the caller (buffers that are idle at the grid barrier).
template <int KG>
__device__ void decide_multi(const Dev& d, const PropParams& pp, int it, long long m, double* s_sum,
                             double* s_key) {
  constexpr int G = 32 * KG;
  const Multi& M = d.mu;
  const int Sp = M.Sp;
  Ctl* ctl = d.ctl;
  __shared__ double s_max[kPropThreads / 32];
  __shared__ unsigned s_gmask;
  __shared__ int s_maxslot;
  if (threadIdx.x == 0) {
    s_gmask = 0;
    s_maxslot = -1;
  }
  const bool pack = M.pack != 0 && KG == 1;
  // thread t sums column t % Sp over the CTAs b = t / Sp (mod Q) with eight
  // independent accumulators; the Q slices are then added in a fixed order
  const int Q = (int)blockDim.x / Sp;
  const int GR = (int)gridDim.x;
  {
    const int jc = threadIdx.x % Sp, q = threadIdx.x / Sp;
    double a[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) a[u] = 0.0;
    if (q < Q)
      for (int b = q; b < GR; b += 8 * Q) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int bb = b + u * Q;
          if (bb < GR) a[u] += __ldcg(M.part + (size_t)bb * Sp + jc);
        }
      }
    s_sum[threadIdx.x] = ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
  }
  __syncthreads();
  double seen = 0.0;
  int live = 0;
  for (int j = threadIdx.x; j < Sp; j += blockDim.x) {
    double L = 0.0;
    for (int q = 0; q < Q; ++q) L += s_sum[q * Sp + j];
    if (j >= M.S) continue;
    const int f = pp.force_iters > 0 ? pp.force_iters : M.force[j];
    if (it == 0) {
      M.col_q[j] = L;
      M.col_last[j] = L;
      M.touched[j] = 0;  // the next offset marks its columns again
      seen = fmax(seen, L);
      if (L == 0.0 && f == 0) {
        M.col_iters[j] = 1;
        M.active[j] = 0;
        if (pack) s_key[j] = -1.0;
      } else {
        M.col_iters[j] = 0;
        M.active[j] = 1;
        live = 1;
        if (pack) s_key[j] = f > 0 ? 1e300 : L;  // forced columns run longest
        else atomicOr(&s_gmask, 1u << (j / G));
      }
    } else if (*(volatile int*)&M.active[j]) {
      M.col_iters[j] = it;
      M.col_last[j] = L;
      seen = fmax(seen, L);
      int stop = f > 0 ? it >= f : L <= pp.eps;
      if (!stop && it >= pp.max_iter) {
        stop = 1;
        ctl->noconv = 1;
      }
      if (stop) {
        M.active[j] = 0;
        // the untaken tail's residual x(k+1) has norm <= (1-c) ||x(k)||_1; L may
        // hold float sums of at most 32 nonnegative terms (relative error below
        // 2^-19), hence the margin
        M.res_bound[j] += (1.0 - ctl->c) * L * (1.0 + 0x1p-18);
      } else {
        live = 1;
        const int slot = pack ? __ldcg(M.col_slot + j) : j;
        atomicOr(&s_gmask, 1u << (slot / G));
        atomicMax(&s_maxslot, slot);
      }
    }
  }
  if (pack && it == 0) {
    // group slots by decreasing ||x(0)||_1 (ties by column), columns without
    // an offset last; a column's slot is its rank
    for (int j = threadIdx.x; j < Sp; j += blockDim.x)
      if (j >= M.S) s_key[j] = -2.0;
    __syncthreads();
    for (int j = threadIdx.x; j < Sp; j += blockDim.x) {
      const double kj = s_key[j];
      int rank = 0;
      for (int i = 0; i < Sp; ++i) {
        const double ki = s_key[i];
        rank += ki > kj || (ki == kj && i < j);
      }
      M.slot_col[rank] = j;
      M.col_slot[j] = rank;
      if (kj >= 0.0) {
        atomicOr(&s_gmask, 1u << (rank / G));
        atomicMax(&s_maxslot, rank);
      }
    }
  }
  seen = warp_max(seen);
  if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = seen;
  const int any = __syncthreads_or(live);
  if (threadIdx.x == 0) {
    double mx = 0.0;
    for (int i = 0; i < kPropWarps; ++i) mx = fmax(mx, s_max[i]);
    if (it < kMaxHist) {
      d.l1_hist[it] = mx;
      d.step_ns[it + 1] = global_ns();
    }
    ctl->iter = it;
    if (it == 0 && !any && kMaxHist > 1) {
      // every x(0) is zero: the do-while's single step is x(1) = 0
      d.l1_hist[1] = 0.0;
      d.step_ns[2] = d.step_ns[1];
      ctl->iter = 1;
    }
    if (it > 0) {
      ctl->visited += m;
      ctl->pull_used = 1;
    }
    int ng = 0;
    for (int g = 0; g < 8; ++g)
      if (s_gmask & (1u << g)) ctl->grp[ng++] = g;
    ctl->n_grp = ng;
    // packed bf16 groups with only slots 0..7 (0..3) running: narrow steps of
    // 8 (4) columns from now on
    ctl->narrow = pack && M.yn0 != nullptr && ng == 1 && ctl->grp[0] == 0 && s_maxslot < 8
                      ? (s_maxslot < 4 ? 4 : 8)
                      : 0;
    ctl->stop = !any;
    for (int i = 0; i < 4; ++i) ctl->ctr[i] = 0;
  }
}

// ---------------------------------------------------------------------------
// Whole-row staging through shared memory. Each warp owns two buffers of
// RingCfg::kRows source rows; a batch of rows of one in-list is copied into a
// buffer by cp.async.bulk (one copy per row, issued by one lane each), and the
// buffer's mbarrier completes once the batch's bytes have landed (transaction
// count = rows x row bytes). The copies need no registers, so many more rows
// are in flight per warp than with register gathers.
// ---------------------------------------------------------------------------
constexpr int kRingBytesPerWarp = 11 * 1024;
constexpr unsigned long long kRingTimeoutNs = 2000000000ull;  // 2 s

template <typename TY, int K>
struct RingCfg {
  static constexpr int kRowBytes = 32 * K * (int)sizeof(TY);  // a multiple of 16
  static constexpr int kFit = kRingBytesPerWarp / (2 * kRowBytes);
  static constexpr int kRows = kFit < 1 ? 1 : (kFit > 32 ? 32 : kFit);
  static constexpr int kBarBytes = 16 * kPropWarps;  // two mbarriers per warp
  static constexpr int kSmem = kBarBytes + kPropWarps * 2 * kRows * kRowBytes;
  // bulk copies need 16-byte aligned addresses and sizes
  static_assert(kRowBytes % 16 == 0 && kBarBytes % 16 == 0, "staged rows must stay 16-byte aligned");
  static_assert(kSmem <= 100 * 1024, "two CTAs per SM must fit with the static shared memory");
};

struct Ring {
  unsigned bar;                 // shared address of the warp's mbarrier 0 (mbarrier 1 follows)
  unsigned rows;                // shared address of the warp's buffer 0 (buffer 1 follows)
  const unsigned char* rows_g;  // the same, as a generic pointer
  unsigned phase;               // bit b: parity of buffer b's next completion
  int buf;                      // the buffer the next batch goes to
};


__device__ __forceinline__ void mbar_init(unsigned a, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(a), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_init_fence() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Arrive (the barrier's one expected arrival) and add `bytes` to the
// transaction count the current phase waits for.
__device__ __forceinline__ void mbar_arrive_expect(unsigned a, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(a), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(unsigned a, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n"
      " .reg .pred p;\n"
      " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n"
      "}"
      : "=r"(ok)
      : "r"(a), "r"(parity)
      : "memory");
  return ok != 0;
}

// Order this thread's generic-proxy accesses to shared memory before later
// async-proxy ones (a bulk copy overwriting rows that were just read).
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void bulk_copy_row(unsigned dst, const void* src, unsigned bytes,
                                              unsigned bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}

// The same with an L2 eviction policy for the source line(s).
__device__ __forceinline__ void bulk_copy_row_pol(unsigned dst, const void* src, unsigned bytes,
                                                  unsigned bar, unsigned long long pol) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], "
      "%2, [%3], %4;" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(bar), "l"(pol)
      : "memory");
}

// Rows u (lane j < cnt holds row j's id) of one column group of the gather
// block (rows of 32 K elements, contiguous: ys is the group's row 0) into
// buffer b.
template <typename TY, int K>
__device__ __forceinline__ void ring_issue(const Ring& rg, int b, int cnt, int u, const TY* ys,
                                           const L2Pol& pol, unsigned long long cold, int hot_n) {
  using C = RingCfg<TY, K>;
  const int lane = threadIdx.x & 31;
  const unsigned bar = rg.bar + 8u * (unsigned)b;
  __syncwarp();  // the warp's reads of buffer b are done ...
  fence_proxy_async_smem();  // ... and come before the copies that overwrite it
  if (lane == 0) mbar_arrive_expect(bar, (unsigned)(cnt * C::kRowBytes));
  __syncwarp();
  if (lane < cnt)
    bulk_copy_row_pol(rg.rows + (unsigned)((b * C::kRows + lane) * C::kRowBytes),
                      ys + (size_t)u * (32 * K), (unsigned)C::kRowBytes, bar,
                      u < hot_n ? pol.keep : cold);
}

// Wait for buffer b's batch. Bounded: after 2 s the call's status becomes
// OSP_ETIMEOUT (the next grid barrier then ends the kernel) and the warp
// waits once more, again bounded, for its copies in flight.
__device__ __forceinline__ void ring_wait(Ring& rg, int b, Ctl* ctl) {
  const unsigned bar = rg.bar + 8u * (unsigned)b;
  const unsigned par = (rg.phase >> b) & 1u;
  if (!mbar_try_wait(bar, par)) {
    const unsigned long long t0 = global_ns();
    unsigned spins = 0;
    while (!mbar_try_wait(bar, par)) {
      if ((++spins & 255u) == 0 && global_ns() - t0 > kRingTimeoutNs) {
        if ((threadIdx.x & 31) == 0) atomicCAS(&ctl->status, 0, (int)OSP_ETIMEOUT);
        const unsigned long long t1 = global_ns();
        while (!mbar_try_wait(bar, par) && global_ns() - t1 < kRingTimeoutNs) {
        }
        break;
      }
    }
  }
  rg.phase ^= 1u << b;
}

// K-element slice of a staged row (plain loads from shared memory).
template <typename T, int K>
__device__ __forceinline__ void load_k(const T* p, T (&out)[K]) {
  constexpr int B = K * (int)sizeof(T);
  if constexpr (B >= 16) {
#pragma unroll
    for (int i = 0; i < B / 16; ++i)
      reinterpret_cast<uint4*>(out)[i] = reinterpret_cast<const uint4*>(p)[i];
  } else if constexpr (B == 8) {
    *reinterpret_cast<uint2*>(out) = *reinterpret_cast<const uint2*>(p);
  } else if constexpr (B == 4) {
    *reinterpret_cast<unsigned*>(out) = *reinterpret_cast<const unsigned*>(p);
  } else {
    *reinterpret_cast<unsigned short*>(out) = *reinterpret_cast<const unsigned short*>(p);
  }
}

// acc += the cnt rows staged in buffer b (this lane's K columns).
template <typename TY, int K, typename A>
__device__ __forceinline__ void ring_sum(const Ring& rg, int b, int cnt, A (&acc)[K]) {
  using C = RingCfg<TY, K>;
  constexpr int Sp = 32 * K;
  const int lane = threadIdx.x & 31;
  const TY* row = reinterpret_cast<const TY*>(rg.rows_g + (size_t)b * C::kRows * C::kRowBytes) +
                  lane * K;
  int j = 0;
  if constexpr (K * sizeof(TY) < 64) {  // four rows at a time while they fit in few registers
    for (; j + 4 <= cnt; j += 4) {
      alignas(16) TY a[4][K];
#pragma unroll
      for (int q = 0; q < 4; ++q) load_k(row + (j + q) * Sp, a[q]);
#pragma unroll
      for (int k = 0; k < K; ++k)
        acc[k] += (to_acc(a[0][k]) + to_acc(a[1][k])) + (to_acc(a[2][k]) + to_acc(a[3][k]));
    }
  } else {
    for (; j + 2 <= cnt; j += 2) {
      alignas(16) TY a[2][K];
#pragma unroll
      for (int q = 0; q < 2; ++q) load_k(row + (j + q) * Sp, a[q]);
#pragma unroll
      for (int k = 0; k < K; ++k) acc[k] += to_acc(a[0][k]) + to_acc(a[1][k]);
    }
  }
  for (; j < cnt; ++j) {
    alignas(16) TY a[K];
    load_k(row + j * Sp, a);
#pragma unroll
    for (int k = 0; k < K; ++k) acc[k] += to_acc(a[k]);
  }
}

// acc += the rows of y over in-list entries p[0 .. L), L >= 1, staged in
// batches of kRows, two batches in flight.
template <typename TY, int K, typename A>
__device__ void ring_sum_list(Ring& rg, const Dev& d, const int* p, int L, const TY* ys,
                              A (&acc)[K], const L2Pol& pol, unsigned long long cold, int hot_n) {
  constexpr int G = RingCfg<TY, K>::kRows;
  const int lane = threadIdx.x & 31;
  auto ids = [&](int s0) -> int {
    const bool in = lane < min(G, L - s0);
    int u = in ? __ldg(p + s0 + lane) : 0;
    if (in && !OSP_GUARD(d.ctl, u >= 0 && u < d.nc, "multi staged piece id", s0, lane, u)) u = 0;
    return u;
  };
  int b = rg.buf;
  ring_issue<TY, K>(rg, b, min(G, L), ids(0), ys, pol, cold, hot_n);
  for (int s0 = 0; s0 < L; s0 += G) {
    if (s0 + G < L) ring_issue<TY, K>(rg, b ^ 1, min(G, L - s0 - G), ids(s0 + G), ys, pol, cold, hot_n);
    ring_wait(rg, b, d.ctl);
    ring_sum<TY, K, A>(rg, b, min(G, L - s0), acc);
    b ^= 1;
  }
  rg.buf = b;
}

// A batch of the staged stream: rows s .. s + cnt - 1 of the in-list of the
// chunk's node lane jc (list at pool_c + off).
struct RowBatch {
  int jc, s, cnt;
  unsigned off;
  bool first, last;
};

}  // namespace

// One CTA: offset items of the changed rows (256 entries of old + new list each).
__global__ void __launch_bounds__(1024) k_offset_multi_plan(Dev d) {
  __shared__ int s_w[32];
  Ctl* ctl = d.ctl;
  if (*(volatile int*)&ctl->status) return;
  const int nr = ctl->n_rec_r;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int per = (nr + 1023) / 1024;
  const int lo = min(nr, tid * per), hi = min(nr, lo + per);
  int mine = 0;
  for (int c = lo; c < hi; ++c) mine += (d.rec_old_len[c] + d.rec_dp[c] + kPiece - 1) / kPiece;
  int x = mine;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_w[w] = x;
  __syncthreads();
  if (w == 0) {
    int t = s_w[lane];
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    s_w[lane] = t;
  }
  __syncthreads();
  int base = (w ? s_w[w - 1] : 0) + x - mine;
  for (int c = lo; c < hi; ++c) {
    const int np = (d.rec_old_len[c] + d.rec_dp[c] + kPiece - 1) / kPiece;
    d.rec_pstart[c] = base;
    for (int q = 0; q < np; ++q) d.piece_rec[base + q] = c;
    base += np;
  }
  if (tid == 0) ctl->n_opieces = s_w[31];
}

// Warp per offset item: R_old[u] times -(1-c)/d_u into xacc over the old
// out-list entries, times +(1-c)/d'_u over the new ones (one combined term
// for an entry in both lists); stamps the targets. Lane l owns columns
// l, l + 32, ..., so each atomic instruction of the warp covers 32
// consecutive columns (8 sectors) of the target's row.
template <int K>
__global__ void __launch_bounds__(256) k_offset_multi(Dev d) {
  constexpr int Sp = 32 * K;
  Ctl* ctl = d.ctl;
  if (*(volatile int*)&ctl->status) return;
  const int np = ctl->n_opieces;
  const double c1 = 1.0 - ctl->c;
  const int epoch = ctl->epoch;
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  unsigned hit = 0;  // bit k: this lane added a nonzero term to its column k
  for (int p = gw; p < np; p += nw) {
    const int c = d.piece_rec[p];
    const int q = p - d.rec_pstart[c];
    const int u = d.rec_r_node[c];
    const int L = d.rec_old_len[c], dp = d.rec_dp[c];
    double ru[K];
#pragma unroll
    for (int k = 0; k < K; ++k) ru[k] = __ldcg(d.mu.r + (size_t)u * Sp + lane + 32 * k);
    bool nz = false;
#pragma unroll
    for (int k = 0; k < K; ++k) nz |= ru[k] != 0.0;
    if (!__any_sync(0xffffffffu, nz)) continue;
    const double wa = L ? c1 / (double)L : 0.0;
    const double wb = dp ? c1 / (double)dp : 0.0;
    const int* oldl = d.pool_r + d.rec_old_off[c];
    const int* newl = d.pool_r + d.rec_fbase[c];
    const int e0 = q * kPiece, e1 = min(e0 + kPiece, L + dp);
    for (int eb = e0; eb < e1; eb += 32) {
      const int e = eb + lane;
      int a = 0;
      double wgt = 0.0;
      if (e < e1) {
        // an entry kept in the new list carries both terms at once:
        // (1-c)(1/d' - 1/d), zero when the degree did not change
        if (e < L) {
          a = oldl[e];
          wgt = contains_i(newl, dp, a) ? wb - wa : -wa;
        } else {
          a = newl[e - L];
          wgt = contains_i(oldl, L, a) ? 0.0 : wb;
        }
      }
      if (!OSP_GUARD(ctl, a >= 0 && a < d.nc, "multi offset target", c, e, a)) a = 0;
      const int cnt = min(32, e1 - eb);
      for (int j = 0; j < cnt; ++j) {
        const double wj = __shfl_sync(0xffffffffu, wgt, j);
        if (wj == 0.0) continue;  // warp-uniform
        const int aj = __shfl_sync(0xffffffffu, a, j);
        double* row = d.mu.xacc + (size_t)aj * Sp + lane;
#pragma unroll
        for (int k = 0; k < K; ++k)
          if (ru[k] != 0.0) {
            atomicAdd(row + 32 * k, wj * ru[k]);
            hit |= 1u << k;
          }
        if (lane == 0) d.mark[aj] = epoch;
      }
    }
  }
  // columns with a nonzero offset entry run this call's steps (the others
  // have x(i) = 0 for every i)
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (hit & (1u << k)) d.mu.touched[lane + 32 * k] = 1;
}

// CPI start for every column: x(0) = c e_{s_j} in column j.
__global__ void k_multi_cpi_begin(Dev d) {
  const Multi& M = d.mu;
  const int j = threadIdx.x;
  if (j < M.S) {
    const int s = M.seeds[j];
    M.xacc[(size_t)s * M.Sp + j] = d.ctl->c;
    M.touched[j] = 1;
    d.mark[s] = d.ctl->epoch;
  }
}

// Column col of R in caller order.
__global__ void k_gather_col(const double* __restrict__ r, int Sp, int col,
                             const int* __restrict__ ext2int, int n, double* out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    out[i] = r[(size_t)ext2int[i] * Sp + col];
}

// CTAs per SM the seed-block kernel is built for: the team gather of bf16
// 32-column groups is built for OSP_TEAM_OCC (default 3; measured 7.3 ms per
// group pass at R-MAT 2^24 against 8.8 ms with 2) CTAs; otherwise three when a
// lane's share of a gather row is at most 4 bytes (few registers), else two.
#ifndef OSP_TEAM_OCC
#define OSP_TEAM_OCC 3
#endif
template <typename TY, int KG>
struct MultiOcc {
  static constexpr int value = std::is_same<TY, __nv_bfloat16>::value && KG == 1
                                   ? OSP_TEAM_OCC
                                   : (KG * (int)sizeof(TY) <= 4 ? 3 : 2);
};

// The seed block, one persistent cooperative launch per call: the x(0) pass
// and every pull step. Columns are processed in groups of G = 32 KG (lane l
// owns columns [KG l, KG l + KG) of the group); a pull step runs each work
// item once per group that still has a running column (an item's groups one
// after the other, so its ids are read from DRAM once; the groups share the
// L2 budget for hot rows), and groups whose columns have all stopped cost
// nothing. The gather blocks (and the
// bf16 residuals) are laid out group-major, [group][node][G], so that a
// group's row is one contiguous slice of G elements; R is [node][Sp].
// kBulk: in-lists stage their source rows in shared memory by bulk
// asynchronous copies (dynamic shared memory RingCfg<TY, KG>::kSmem); else
// each lane gathers its columns of up to kDepth rows into registers.
template <typename TY, int KG, bool kBulk>
__global__ void __launch_bounds__(kPropThreads, MultiOcc<TY, KG>::value)
    k_propagate_multi(Dev d, PropParams pp) {
  using A = typename AccOf<TY>::type;
  constexpr int G = 32 * KG;
  constexpr bool FB = Feedback<TY>::on;
  // bf16 rows of 32-column groups are gathered by teams of 8 lanes over a flat
  // edge stream (team_stream / team_piece); the other forms walk node by node
  constexpr bool kTeam = std::is_same<TY, __nv_bfloat16>::value && KG == 1 && !kBulk;
  __shared__ __align__(16) float s_team_acc[kTeam ? kPropWarps * 1024 : 1];  // node x column sums
  __shared__ __align__(16) __nv_bfloat16 s_team_e[kTeam ? kPropWarps * 1024 : 8];  // residual rows
  __shared__ BarShared sh;
  __shared__ double s_part[kMaxSeeds];  // per column |x| sums of the CTA (shared-memory atomics)
  // the decision's scratch: the team node sums (idle at the grid barrier), else its own
  __shared__ double s_dec_own[kTeam ? 1 : kPropThreads + kMaxSeeds];
  double* s_dec = kTeam ? reinterpret_cast<double*>(s_team_acc) : s_dec_own;
  __shared__ int s_grp[8];
  __shared__ int s_ngrp;
  __shared__ unsigned s_tmask;
  extern __shared__ __align__(128) unsigned char dsm[];
  Ctl* ctl = d.ctl;
  if (*(volatile int*)&ctl->status) return;
  Ring rg{};
  if constexpr (kBulk) {
    using C = RingCfg<TY, KG>;
    const int w = threadIdx.x >> 5;
    rg.bar = smem_u32(dsm) + 16u * (unsigned)w;
    const int off = C::kBarBytes + w * 2 * C::kRows * C::kRowBytes;
    rg.rows = smem_u32(dsm) + (unsigned)off;
    rg.rows_g = dsm + off;
    if ((threadIdx.x & 31) == 0) {
      mbar_init(rg.bar, 1);
      mbar_init(rg.bar + 8u, 1);
      mbar_init_fence();
    }
    __syncthreads();
  }
  const Multi& M = d.mu;
  const int Sp = M.Sp;
  // packed groups (bf16 team path): group slot q holds column slot_col[q],
  // chosen per call by the x(0) decision so that columns likely to run long
  // share groups; R, the offsets and the per-column state stay by column
  const bool pack = kTeam && M.pack != 0;
  const size_t gs = (size_t)d.nc * G;  // gather block: elements per column group
  const int n = ctl->n;
  const long long m = ctl->m;
  const int epoch = ctl->epoch;
  const int n_hubs = ctl->n_hubs;
  const int n_pieces = ctl->n_pieces;
  const int n_tasks = ctl->n_tasks;
  const int hub_thr = ctl->hub_thr, hub_piece = ctl->hub_piece;
  const L2Pol pol = make_l2pol();
  const int hot_n = pp.hot_n;
  const unsigned long long cold = hot_n > 0 ? pol.once : pol.normal;
  TY* yb[2] = {(TY*)M.y0, (TY*)M.y1};
  TY* eb = (TY*)M.e;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  double* my_part = s_part;
  if (blockIdx.x == 0 && threadIdx.x == 0) d.step_ns[0] = global_ns();

  // per-CTA column sums of the warps' partials (fixed order) into M.part
  auto column_sums = [&]() {
    __syncthreads();
    for (int j = threadIdx.x; j < Sp; j += blockDim.x) {
      double a = 0.0;
      a = s_part[j];
      M.part[(size_t)blockIdx.x * Sp + j] = a;
    }
    __threadfence();
  };

  // x(0): stamped rows move from xacc into R and, scaled, into y(0); every
  // node with out-edges gets its y(0) row (zero when not stamped) in each
  // column group that has a nonzero offset entry
  if (pack) {
    // 1. ||x(0)||_1 per column from the stamped rows; the decision orders the
    //    columns by it (largest first: a larger offset needs more steps) into
    //    group slots and picks the groups that hold a running column
    for (int j = lane; j < Sp; j += 32) my_part[j] = 0.0;
    unsigned tb = 0;  // bit k: column lane + 32 k has an offset entry
    for (int k = 0; k < 8 && lane + 32 * k < M.S; ++k)
      if (*(volatile int*)&M.touched[lane + 32 * k]) tb |= 1u << k;
    __syncthreads();
    for (int vb = gw * 32; vb < n && __any_sync(0xffffffffu, tb != 0); vb += nw * 32) {
      const int vl = vb + lane;
      unsigned stamped = __ballot_sync(0xffffffffu, vl < n && __ldcg(d.mark + vl) == epoch);
      while (stamped) {
        const int v = vb + __ffs(stamped) - 1;
        stamped &= stamped - 1;
        for (unsigned t = tb; t; t &= t - 1) {
          const int j = lane + 32 * (__ffs(t) - 1);
          atomicAdd(my_part + j, fabs(__ldcg(M.xacc + (size_t)v * Sp + j)));
        }
      }
    }
    column_sums();
    if (bar_arrive(ctl, sh)) decide_multi<KG>(d, pp, 0, m, s_dec, s_dec + kPropThreads);
    if (!bar_release(ctl, sh)) return;
    // 2. R += x(0) and the y(0) rows, in group slots
    if (threadIdx.x < 8) s_grp[threadIdx.x] = *(volatile int*)&ctl->grp[threadIdx.x];
    if (threadIdx.x == 0) s_ngrp = *(volatile int*)&ctl->n_grp;
    __syncthreads();
    const int ng = s_ngrp;
    int colg[8];
    unsigned actg = 0;  // bit gi: this lane's column of group s_grp[gi] runs
#pragma unroll
    for (int gi = 0; gi < 8; ++gi) {
      colg[gi] = 0;
      if (gi < ng) {
        colg[gi] = __ldcg(M.slot_col + s_grp[gi] * G + lane);
        if (*(volatile int*)&M.active[colg[gi]]) actg |= 1u << gi;
      }
    }
    for (int vb = gw * 32; vb < n && ng > 0; vb += nw * 32) {
      const int vl = vb + lane;
      const unsigned stamped = __ballot_sync(0xffffffffu, vl < n && __ldcg(d.mark + vl) == epoch);
      const A s_l = vl < n ? scale_of<A>(d, vl) : (A)0;
      unsigned work = stamped | __ballot_sync(0xffffffffu, s_l != (A)0);
      while (work) {
        const int jj = __ffs(work) - 1;
        work &= work - 1;
        const int v = vb + jj;
        const bool st = (stamped >> jj) & 1u;
        const A s = __shfl_sync(0xffffffffu, s_l, jj);
#pragma unroll
        for (int gi = 0; gi < 8; ++gi) {
          if (gi >= ng || !((actg >> gi) & 1u)) continue;
          const size_t ybase = s_grp[gi] * gs + (size_t)v * G + lane;
          TY yv = from_acc((A)0, (TY*)nullptr), ev = yv;
          if (st) {
            const size_t rb = (size_t)v * Sp + colg[gi];
            const double x = __ldcg(M.xacc + rb);
            if (x != 0.0) {
              M.r[rb] += x;
              M.xacc[rb] = 0.0;
              const A w = (A)((A)x * s);
              yv = from_acc(w, (TY*)nullptr);
              if constexpr (FB) ev = __float2bfloat16_rn(w - __bfloat162float(yv));
            }
          }
          if (s != (A)0) {
            const TY y1[1] = {yv}, e1[1] = {ev};
            st_pol(yb[0] + ybase, y1, pol.once);
            if constexpr (FB) st_pol(eb + ybase, e1, pol.once);
          }
        }
      }
    }
    if (bar_arrive(ctl, sh) && threadIdx.x == 0) ctl->ctr[1] = 0;
    if (!bar_release(ctl, sh)) return;
  } else {
    if (threadIdx.x == 0) s_tmask = 0;
    for (int j = lane; j < Sp; j += 32) my_part[j] = 0.0;
    __syncthreads();
    for (int j = threadIdx.x; j < Sp && j < M.S; j += blockDim.x)
      if (*(volatile int*)&M.touched[j]) atomicOr(&s_tmask, 1u << (j / G));
    __syncthreads();
    const unsigned tmask = s_tmask;
    unsigned lane_touch = 0;  // bit g: one of this lane's columns in group g has an offset entry
    for (unsigned tm = tmask; tm; tm &= tm - 1) {
      const int g = __ffs(tm) - 1;
      for (int k = 0; k < KG; ++k) {
        const int j = g * G + lane * KG + k;
        if (j < M.S && *(volatile int*)&M.touched[j]) lane_touch |= 1u << g;
      }
    }
    for (int vb = gw * 32; vb < n && tmask; vb += nw * 32) {
      const int vl = vb + lane;
      const unsigned stamped = __ballot_sync(0xffffffffu, vl < n && __ldcg(d.mark + vl) == epoch);
      const A s_l = vl < n ? scale_of<A>(d, vl) : (A)0;
      unsigned work = stamped | __ballot_sync(0xffffffffu, s_l != (A)0);
      while (work) {
        const int jj = __ffs(work) - 1;
        work &= work - 1;
        const int v = vb + jj;
        const bool st = (stamped >> jj) & 1u;
        const A s = __shfl_sync(0xffffffffu, s_l, jj);
        for (unsigned tm = tmask; tm; tm &= tm - 1) {
          const int g = __ffs(tm) - 1;
          if (!((lane_touch >> g) & 1u)) continue;  // none of this lane's columns has an offset
          const size_t rbase = (size_t)v * Sp + g * G + lane * KG;
          const size_t ybase = g * gs + (size_t)v * G + lane * KG;
          alignas(16) TY yv[KG];
          alignas(16) TY ev[KG];
          if (st) {
            alignas(16) double x[KG], rr[KG], z[KG];
            ld_pol(M.xacc + rbase, x, pol.once);
            ld_pol(M.r + rbase, rr, pol.once);
#pragma unroll
            for (int k = 0; k < KG; ++k) {
              rr[k] += x[k];
              atomicAdd(my_part + g * G + lane * KG + k, fabs(x[k]));
              z[k] = 0.0;
              const A w = (A)((A)x[k] * s);
              yv[k] = from_acc(w, (TY*)nullptr);
              if constexpr (FB) ev[k] = __float2bfloat16_rn(w - __bfloat162float(yv[k]));
            }
            st_pol(M.r + rbase, rr, pol.once);
            st_pol(M.xacc + rbase, z, pol.once);
          } else {
#pragma unroll
            for (int k = 0; k < KG; ++k) {
              yv[k] = from_acc((A)0, (TY*)nullptr);
              ev[k] = yv[k];
            }
          }
          if (s != (A)0) {
            st_pol(yb[0] + ybase, yv, pol.once);
            if constexpr (FB) st_pol(eb + ybase, ev, pol.once);
          }
        }
      }
    }
    column_sums();
    if (bar_arrive(ctl, sh)) decide_multi<KG>(d, pp, 0, m, s_dec, s_dec + kPropThreads);
    if (!bar_release(ctl, sh)) return;
  }

  A* hub_acc = (A*)M.hub_acc;
  int prev_narrow = 0;  // row width of the compact block the last step wrote (0: none)
  for (int it = 1;; ++it) {
    if (*(volatile int*)&ctl->stop) break;
    if (threadIdx.x < 8) s_grp[threadIdx.x] = *(volatile int*)&ctl->grp[threadIdx.x];
    if (threadIdx.x == 0) s_ngrp = *(volatile int*)&ctl->n_grp;
    for (int j = lane; j < Sp; j += 32) my_part[j] = 0.0;
    __syncthreads();
    const TY* ys = yb[(it - 1) & 1];
    TY* yd = yb[it & 1];
    const int n_items = n_pieces + n_tasks;
    const long long total = (long long)s_ngrp * n_items;
    // the groups of a step are gathered side by side: they share the L2
    // budget for hot rows
    const int hot_step = s_ngrp > 1 ? hot_n / s_ngrp : hot_n;
    int cur = -1;  // column group of the items this warp works on now
    int pcol = -1;  // packed bf16 groups: this lane's column in group cur
    unsigned act = 0;
    bool on4 = false;
    double l1[KG];
#pragma unroll
    for (int k = 0; k < KG; ++k) l1[k] = 0.0;
    auto flush = [&]() {
      if (cur >= 0) {
#pragma unroll
        for (int k = 0; k < KG; ++k) {
          atomicAdd(my_part + (kTeam && pack ? pcol : cur * G + lane * KG) + k, l1[k]);
          l1[k] = 0.0;
        }
      }
    };
    int narrow = 0;  // row width of a narrow step (0: a step over column groups)
    if constexpr (kTeam) narrow = *(volatile int*)&ctl->narrow;
    if constexpr (kTeam) {
      if (narrow) {
        __nv_bfloat16* yn[2] = {(__nv_bfloat16*)M.yn0, (__nv_bfloat16*)M.yn1};
        const __nv_bfloat16* src =
            prev_narrow ? yn[(it - 1) & 1] : reinterpret_cast<const __nv_bfloat16*>(ys);
        const int stride = prev_narrow ? prev_narrow : 32;
        float* acc_s = s_team_acc + wid * 1024;
        if (narrow == 4) {
          Narrow<4> N{src, stride, yn[it & 1], reinterpret_cast<__nv_bfloat16*>(eb), {}, 0u};
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            N.col[c] = __ldcg(M.slot_col + c);
            if (*(volatile int*)&M.active[N.col[c]]) N.act |= 1u << c;
          }
          narrow_step<4>(d, M, N, n_items, n_pieces, hub_thr, hub_piece, (float*)hub_acc, acc_s,
                         my_part, ctl);
        } else {
          Narrow<8> N{src, stride, yn[it & 1], reinterpret_cast<__nv_bfloat16*>(eb), {}, 0u};
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            N.col[c] = __ldcg(M.slot_col + c);
            if (*(volatile int*)&M.active[N.col[c]]) N.act |= 1u << c;
          }
          narrow_step<8>(d, M, N, n_items, n_pieces, hub_thr, hub_piece, (float*)hub_acc, acc_s,
                         my_part, ctl);
        }
      }
    }
    prev_narrow = narrow;
    if (!narrow)
    for (int k = 0;; ++k) {
      int t = gw;  // the first item is the warp's own number, later ones come from the counter
      if (k > 0) {
        if (total <= nw) break;
        if (lane == 0) t = nw + atomicAdd(&ctl->ctr[1], 1);
        t = __shfl_sync(0xffffffffu, t, 0);
      }
      if (t >= total) break;
      // task-major: a work item's groups come one after the other, so its
      // in-list ids and node headers are read from DRAM once for all groups
      const int gi = t % s_ngrp;
      const int ti = t / s_ngrp;
      const int g = s_grp[gi];
      if (g != cur) {
        flush();
        cur = g;
        act = 0;
        if constexpr (kTeam) pcol = pack ? __ldcg(M.slot_col + g * G + lane) : g * G + lane;
#pragma unroll
        for (int k = 0; k < KG; ++k)
          act |= (unsigned)(*(volatile int*)&M.active[(kTeam ? pcol : g * G + lane * KG) + k] != 0)
                 << k;
        if constexpr (kTeam) {
          // team gathers: lane (t, s) loads columns [4 s, 4 s + 4) of a row
          const unsigned am = __ballot_sync(0xffffffffu, act != 0);
          on4 = ((am >> (4 * (lane & 7))) & 0xFu) != 0;
        }
      }
      const TY* ysg = ys + g * gs;           // the group's gather rows, G elements apart
      const TY* ysl = ysg + lane * KG;       // this lane's columns of them
      const size_t c0 = (size_t)g * G + lane * KG;  // slot: gather rows, residuals, hub sums
      const size_t rc0 = kTeam ? (size_t)pcol : c0;  // column of R
      auto rbase_of = [&](int v) { return (size_t)v * Sp + rc0; };
      auto ybase_of = [&](int v) { return g * gs + (size_t)v * G + lane * KG; };
      if (ti < n_pieces) {
        // a piece of a long in-list; the piece that completes the list finishes it
        const int h = __ldg(d.piece_hub + ti);
        const int v = __ldg(d.hubs + h);
        const int piece = ti - __ldg(d.hub_pstart + h);
        const int full = __ldg(d.len_c + v);
        const int* p = d.pool_c + __ldg(d.off_c + v) + (unsigned)(piece * hub_piece);
        const int L = min(hub_piece, full - piece * hub_piece);
        if constexpr (kTeam) {
          float a4[4];
          team_piece(p, L, ysg, on4, pol, cold, hot_step, a4);
          float* ha4 = (float*)hub_acc + (size_t)h * Sp + (size_t)g * G + 4 * lane;
          if (lane < 8 && on4) {
#pragma unroll
            for (int c = 0; c < 4; ++c) atomicAdd(ha4 + c, a4[c]);
          }
          __threadfence();
          int last = 0;
          if (lane == 0) {
            const int np = (full + hub_piece - 1) / hub_piece;
            last = atomicAdd(&M.hub_cnt[h * 8 + g], 1) == np - 1;
          }
          last = __shfl_sync(0xffffffffu, last, 0);
          if (last) {
            __threadfence();
            float* hx = (float*)hub_acc + (size_t)h * Sp + c0;  // lane = column
            const float x = __ldcg(hx);
            *hx = 0.f;
            if (lane == 0) M.hub_cnt[h * 8 + g] = 0;
            const float sv = scale_of<float>(d, v);
            if (act) {
              red_add_once(M.r + rbase_of(v), (double)x, pol.once);
              l1[0] += fabs((double)x);
              if (sv != 0.f) {
                const float w = x * sv + __bfloat162float(eb[ybase_of(v)]);
                const __nv_bfloat16 yv = __float2bfloat16_rn(w);
                yd[ybase_of(v)] = yv;
                eb[ybase_of(v)] = __float2bfloat16_rn(w - __bfloat162float(yv));
              }
            }
          }
          continue;
        }
        A acc[KG];
#pragma unroll
        for (int k = 0; k < KG; ++k) acc[k] = (A)0;
        if constexpr (kBulk) ring_sum_list<TY, KG, A>(rg, d, p, L, ysg, acc, pol, cold, hot_n);
        else sum_rows<TY, KG, A>(p, L, ysl, G, acc, -1, pol, cold, hot_n, act != 0);
        A* ha = hub_acc + (size_t)h * Sp + c0;
#pragma unroll
        for (int k = 0; k < KG; ++k) atomicAdd(ha + k, acc[k]);
        __threadfence();
        int last = 0;
        if (lane == 0) {
          const int np = (full + hub_piece - 1) / hub_piece;
          last = atomicAdd(&M.hub_cnt[h * 8 + g], 1) == np - 1;
        }
        last = __shfl_sync(0xffffffffu, last, 0);
        if (last) {
          __threadfence();
#pragma unroll
          for (int k = 0; k < KG; ++k) {
            acc[k] = __ldcg(ha + k);
            ha[k] = (A)0;
          }
          if (lane == 0) M.hub_cnt[h * 8 + g] = 0;
          const A s = scale_of<A>(d, v);
          alignas(16) double rr[KG];
          alignas(16) TY eo[KG];
#pragma unroll
          for (int k = 0; k < KG; ++k) eo[k] = from_acc((A)0, (TY*)nullptr);
          if (act) {
            ld_pol(M.r + rbase_of(v), rr, pol.once);
            if (FB && s != (A)0) ld_pol(eb + ybase_of(v), eo, pol.once);
          }
          finish_slice<TY, KG, A>(M, rbase_of(v), ybase_of(v), acc, s, true, rr, eo, act, yd, l1, pol);
        }
        continue;
      }
      const int task = ti - n_pieces;
      const int c0t = __ldg(d.task_first + task), c1t = __ldg(d.task_first + task + 1);
      if constexpr (kTeam) {
        float* acc_s = s_team_acc + wid * 1024;
        __nv_bfloat16* e_s = s_team_e + wid * 1024;
        // list lengths, offsets and scales of the next run of 32 nodes load
        // while the current run is summed
        int nx_len = 0;
        unsigned nx_off = 0;
        float nx_s = 0.f;
        auto header = [&](int vb) {
          const int vl = vb + lane;
          nx_len = 0;
          nx_off = 0;
          nx_s = 0.f;
          if (vl < c1t) {
            nx_len = __ldg(d.len_c + vl);
            nx_off = __ldg(d.off_c + vl);
            nx_s = scale_of<float>(d, vl);
          }
        };
        header(c0t);
        for (int vb = c0t; vb < c1t; vb += 32) {
          const int vl = vb + lane;
          const int my_len = nx_len;
          const unsigned my_off = nx_off;
          const float my_s = nx_s;
          if (vb + 32 < c1t) header(vb + 32);
          const bool mine = vl < c1t && my_len <= hub_thr;  // hubs go by pieces
          const unsigned fin = __ballot_sync(0xffffffffu, mine && (my_len > 0 || my_s != 0.f));
          if (!fin) continue;
          // this node's residual row (all 32 columns) into shared memory, in flight
          // while the stream runs
          if (((fin >> lane) & 1u) && my_s != 0.f) {
            const __nv_bfloat16* er = eb + g * gs + (size_t)vl * G;
#pragma unroll
            for (int q = 0; q < 4; ++q) cp_async16(e_s + lane * 32 + 8 * q, er + 8 * q);
          }
#pragma unroll
          for (int q = 0; q < 8; ++q)
            reinterpret_cast<float4*>(acc_s)[lane + 32 * q] = make_float4(0.f, 0.f, 0.f, 0.f);
          __syncwarp();
          team_stream(d.pool_c, mine ? my_len : 0, my_off, ysg, on4, pol, cold, hot_step, acc_s);
          cp_async_wait_all();
          __syncwarp();
          // finish: lane = column; |x| of the run summed in float (at most 32
          // nonnegative terms), then added to the FP64 partial once
          float l1f = 0.f;
          for (unsigned fb = fin; fb; fb &= fb - 1) {
            const int j = __ffs(fb) - 1;
            const int v = vb + j;
            const float sj = __shfl_sync(0xffffffffu, my_s, j);
            const bool has_in = __shfl_sync(0xffffffffu, my_len, j) > 0;
            if (!act) continue;
            const float x = acc_s[j * 32 + lane];
            if (has_in) {
              red_add_once(M.r + rbase_of(v), (double)x, pol.once);
              l1f += fabsf(x);
            }
            if (sj != 0.f) {
              const float w = x * sj + __bfloat162float(e_s[j * 32 + lane]);
              const __nv_bfloat16 yv = __float2bfloat16_rn(w);
              yd[ybase_of(v)] = yv;
              eb[ybase_of(v)] = __float2bfloat16_rn(w - __bfloat162float(yv));
            }
          }
          l1[0] += (double)l1f;
          __syncwarp();
        }
        continue;
      }
      for (int vb = c0t; vb < c1t; vb += 32) {
        // offsets, lengths and scales of up to 32 consecutive nodes, coalesced
        const int vl = vb + lane;
        int my_len = 0;
        unsigned my_off = 0;
        A my_s = (A)0;
        if (vl < c1t) {
          my_len = __ldg(d.len_c + vl);
          my_off = __ldg(d.off_c + vl);
          my_s = scale_of<A>(d, vl);
        }
        const int cnt = min(32, c1t - vb);
        // a node with an in-list adds x(i) into R; a node with out-edges writes
        // its next gather row (zero, or the carried residual, without in-list)
        unsigned todo = __ballot_sync(0xffffffffu, lane < cnt && my_len <= hub_thr &&
                                                       (my_len > 0 || my_s != (A)0));
        if (!todo) continue;
        if constexpr (kBulk) {
          // batches of up to kRows rows of one in-list, nodes in order: the next
          // batch's copies and the ids of the one after are in flight while a
          // batch is summed; a node's row of R loads with its first batch
          constexpr int GR = RingCfg<TY, KG>::kRows;
          int pj = 0, plen = 0, ps = 0;
          unsigned poff = 0;
          // nodes without in-list: their gather row only
          unsigned empty = todo & __ballot_sync(0xffffffffu, my_len == 0);
          todo &= ~empty;
          while (empty) {
            const int jj = __ffs(empty) - 1;
            empty &= empty - 1;
            const int v = vb + jj;
            const A s = __shfl_sync(0xffffffffu, my_s, jj);
            A acc[KG];
            alignas(16) double rr[KG];
            alignas(16) TY eo[KG];
#pragma unroll
            for (int k = 0; k < KG; ++k) {
              acc[k] = (A)0;
              rr[k] = 0.0;
              eo[k] = from_acc((A)0, (TY*)nullptr);
            }
            if (FB && act) ld_pol(eb + ybase_of(v), eo, pol.once);
            finish_slice<TY, KG, A>(M, rbase_of(v), ybase_of(v), acc, s, false, rr, eo, act, yd, l1, pol);
          }
          if (!todo) continue;
          auto next = [&](RowBatch& o) -> bool {
            if (ps >= plen) {
              if (!todo) return false;
              pj = __ffs(todo) - 1;
              todo &= todo - 1;
              plen = __shfl_sync(0xffffffffu, my_len, pj);
              poff = __shfl_sync(0xffffffffu, my_off, pj);
              ps = 0;
            }
            o.jc = pj;
            o.off = poff;
            o.s = ps;
            o.cnt = min(GR, plen - ps);
            o.first = ps == 0;
            o.last = ps + GR >= plen;
            ps += GR;
            return true;
          };
          auto ids_of = [&](const RowBatch& o) -> int {
            int u = lane < o.cnt ? __ldg(d.pool_c + o.off + (unsigned)(o.s + lane)) : 0;
            if (lane < o.cnt && !OSP_GUARD(ctl, u >= 0 && u < d.nc, "multi staged id", o.jc, o.s, u))
              u = 0;
            return u;
          };
          RowBatch b0, b1, b2;
          next(b0);
          ring_issue<TY, KG>(rg, rg.buf, b0.cnt, ids_of(b0), ysg, pol, cold, hot_n);
          alignas(16) double rr_n[KG];
          alignas(16) TY eo_n[KG];
#pragma unroll
          for (int k = 0; k < KG; ++k) rr_n[k] = 0.0;
          if (act) ld_pol(M.r + rbase_of(vb + b0.jc), rr_n, pol.once);
          A s_n = __shfl_sync(0xffffffffu, my_s, b0.jc);
#pragma unroll
          for (int k = 0; k < KG; ++k) eo_n[k] = from_acc((A)0, (TY*)nullptr);
          if (FB && act && s_n != (A)0) ld_pol(eb + ybase_of(vb + b0.jc), eo_n, pol.once);
          bool h1 = next(b1);
          int u1 = h1 ? ids_of(b1) : 0;
          alignas(16) double rr[KG];
          alignas(16) TY eo[KG];
          A s = (A)0;
          A acc[KG];
#pragma unroll
          for (int k = 0; k < KG; ++k) acc[k] = (A)0;
          for (;;) {
            if (b0.first) {
#pragma unroll
              for (int k = 0; k < KG; ++k) {
                rr[k] = rr_n[k];
                eo[k] = eo_n[k];
                acc[k] = (A)0;
              }
              s = s_n;
            }
            const int b = rg.buf;
            if (h1) {
              ring_issue<TY, KG>(rg, b ^ 1, b1.cnt, u1, ysg, pol, cold, hot_n);
              if (b1.first) {
                if (act) ld_pol(M.r + rbase_of(vb + b1.jc), rr_n, pol.once);
                s_n = __shfl_sync(0xffffffffu, my_s, b1.jc);
                if (FB && act && s_n != (A)0) ld_pol(eb + ybase_of(vb + b1.jc), eo_n, pol.once);
              }
            }
            const bool h2 = h1 && next(b2);
            const int u2 = h2 ? ids_of(b2) : 0;
            ring_wait(rg, b, ctl);
            ring_sum<TY, KG, A>(rg, b, b0.cnt, acc);
            if (b0.last)
              finish_slice<TY, KG, A>(M, rbase_of(vb + b0.jc), ybase_of(vb + b0.jc), acc, s, true,
                                      rr, eo, act, yd, l1, pol);
            if (!h1) break;
            rg.buf = b ^ 1;
            b0 = b1;
            b1 = b2;
            h1 = h2;
            u1 = u2;
          }
          continue;
        }
        int jn = __ffs(todo) - 1;
        todo &= todo - 1;
        int len_n = __shfl_sync(0xffffffffu, my_len, jn);
        unsigned off_n = __shfl_sync(0xffffffffu, my_off, jn);
        A s_n = __shfl_sync(0xffffffffu, my_s, jn);
        int idx_n = lane < len_n ? __ldg(d.pool_c + off_n + lane) : 0;
        alignas(16) double rr_n[KG];
        alignas(16) TY eo_n[KG];
#pragma unroll
        for (int k = 0; k < KG; ++k) {
          rr_n[k] = 0.0;
          eo_n[k] = from_acc((A)0, (TY*)nullptr);
        }
        if (act && len_n > 0) ld_pol(M.r + rbase_of(vb + jn), rr_n, pol.once);
        if (FB && act && s_n != (A)0) ld_pol(eb + ybase_of(vb + jn), eo_n, pol.once);
        for (;;) {
          const int jc = jn, len = len_n;
          const unsigned off = off_n;
          const int idx = idx_n;
          const A s = s_n;
          alignas(16) double rr[KG];
          alignas(16) TY eo[KG];
#pragma unroll
          for (int k = 0; k < KG; ++k) {
            rr[k] = rr_n[k];
            eo[k] = eo_n[k];
          }
          const bool more = todo != 0;
          if (more) {
            jn = __ffs(todo) - 1;
            todo &= todo - 1;
            len_n = __shfl_sync(0xffffffffu, my_len, jn);
            off_n = __shfl_sync(0xffffffffu, my_off, jn);
            s_n = __shfl_sync(0xffffffffu, my_s, jn);
            idx_n = lane < len_n ? __ldg(d.pool_c + off_n + lane) : 0;
            if (act && len_n > 0) ld_pol(M.r + rbase_of(vb + jn), rr_n, pol.once);
            if (FB && act && s_n != (A)0) ld_pol(eb + ybase_of(vb + jn), eo_n, pol.once);
          }
          const int v = vb + jc;
          A acc[KG];
#pragma unroll
          for (int k = 0; k < KG; ++k) acc[k] = (A)0;
          if (len > 0)
            sum_rows<TY, KG, A>(d.pool_c + off, len, ysl, G, acc, idx, pol, cold, hot_n, act != 0);
          finish_slice<TY, KG, A>(M, rbase_of(v), ybase_of(v), acc, s, len > 0, rr, eo, act, yd, l1, pol);
          if (!more) break;
        }
      }
    }
    flush();
    column_sums();
    if (bar_arrive(ctl, sh)) decide_multi<KG>(d, pp, it, m, s_dec, s_dec + kPropThreads);
    if (!bar_release(ctl, sh)) return;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) ctl->epoch = epoch + 1;
}

namespace {

struct MultiFn {
  const void* fn;
  int smem;  // dynamic shared memory bytes
};

template <typename TY, int KG>
MultiFn multi_fn_k(bool bulk) {
  if (bulk) return {(const void*)k_propagate_multi<TY, KG, true>, RingCfg<TY, KG>::kSmem};
  return {(const void*)k_propagate_multi<TY, KG, false>, 0};
}

template <typename TY>
MultiFn multi_fn(int KG, bool bulk) {
  switch (KG) {
    case 1: return multi_fn_k<TY, 1>(bulk);
    case 2: return multi_fn_k<TY, 2>(bulk);
    case 4: return multi_fn_k<TY, 4>(bulk);
    default: return multi_fn_k<TY, 8>(bulk);
  }
}

MultiFn pick_multi(int precision, int KG, bool bulk) {
  if (precision == OSP_PREC_FP64) return multi_fn<double>(KG, bulk);
  if (precision == OSP_PREC_FP32_ACC64) return multi_fn<float>(KG, bulk);
  return multi_fn<__nv_bfloat16>(KG, bulk);
}

}  // namespace

int propagate_multi_grid(int precision, int KG, int num_sms, bool bulk) {
  const MultiFn f = pick_multi(precision, KG, bulk);
  if (f.smem > 0 &&
      cudaFuncSetAttribute(f.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, f.smem) != cudaSuccess)
    return 0;
  int bps = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, f.fn, kPropThreads, f.smem) != cudaSuccess ||
      bps <= 0)
    return 0;
  bps = bps > 4 ? 4 : bps;
  const int g = bps * num_sms;
  return g > kMaxGrid ? kMaxGrid : g;
}

cudaError_t launch_propagate_multi(const Dev& d, const PropParams& pp, int precision, int KG,
                                   int grid, bool bulk, cudaStream_t s) {
  Dev dd = d;
  PropParams p = pp;
  void* args[] = {&dd, &p};
  const MultiFn f = pick_multi(precision, KG, bulk);
  return cudaLaunchCooperativeKernel(f.fn, dim3(grid), dim3(kPropThreads), args, (size_t)f.smem, s);
}

// ---------------------------------------------------------------------------
// Failure-detection self-tests: the bounded waits of the persistent kernels
// are made to run out on purpose (a CTA that never arrives; an mbarrier whose
// announced bytes never all land), and the status word must report it.
// ---------------------------------------------------------------------------
__global__ void k_selftest_barrier(Ctl* ctl, int lose) {
  __shared__ BarShared sh;
  if (lose && blockIdx.x == 0) return;  // this CTA never arrives
  if (bar_arrive(ctl, sh) && threadIdx.x == 0) ctl->iter = 1;
  bar_release(ctl, sh);
}

__global__ void k_selftest_stage(Ctl* ctl, const float* src, int lose) {
  using C = RingCfg<float, 1>;
  extern __shared__ __align__(128) unsigned char dsm[];
  Ring rg{};
  rg.bar = smem_u32(dsm);
  rg.rows = smem_u32(dsm) + C::kBarBytes;
  rg.rows_g = dsm + C::kBarBytes;
  if (threadIdx.x == 0) {
    mbar_init(rg.bar, 1);
    mbar_init(rg.bar + 8u, 1);
    mbar_init_fence();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    // two rows announced; with `lose` only the first is copied
    mbar_arrive_expect(rg.bar, 2u * C::kRowBytes);
    bulk_copy_row(rg.rows, src, C::kRowBytes, rg.bar);
    if (!lose) bulk_copy_row(rg.rows + C::kRowBytes, src + 32, C::kRowBytes, rg.bar);
  }
  __syncwarp();
  ring_wait(rg, 0, ctl);
  if (threadIdx.x == 0 && *(volatile int*)&ctl->status == 0) {
    const float* r = reinterpret_cast<const float*>(rg.rows_g);
    ctl->iter = (r[0] == src[0] && r[63] == src[63]) ? 1 : 2;  // both rows arrived intact
  }
}

cudaError_t launch_selftest(Ctl* ctl, const float* src, int which, int lose, cudaStream_t s) {
  if (which == 0) {
    k_selftest_barrier<<<4, 64, 0, s>>>(ctl, lose);
  } else {
    k_selftest_stage<<<1, 32, RingCfg<float, 1>::kBarBytes + 2 * RingCfg<float, 1>::kRowBytes, s>>>(
        ctl, src, lose);
  }
  return cudaGetLastError();
}

cudaError_t launch_offset_multi(const Dev& d, int grid, cudaStream_t s) {
  switch (d.mu.K) {
    case 1: k_offset_multi<1><<<grid, 256, 0, s>>>(d); break;
    case 2: k_offset_multi<2><<<grid, 256, 0, s>>>(d); break;
    case 4: k_offset_multi<4><<<grid, 256, 0, s>>>(d); break;
    default: k_offset_multi<8><<<grid, 256, 0, s>>>(d); break;
  }
  return cudaGetLastError();
}

}  // namespace osp
