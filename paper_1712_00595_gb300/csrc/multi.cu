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
//            rows through per-warp rings in shared memory (k_propagate_ring) or
//            a warp per node, lanes over columns (k_propagate_multi); long
//            in-lists in pieces.
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

// K contiguous elements (K * sizeof(T) bytes, naturally aligned).
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
  // rows gathered per batch of loads (more when a lane's share is small)
  static constexpr int kDepth = KG * (int)sizeof(TY) <= 8 ? 16 : 8;
};

// Sum of the gather rows of in-list entries p[0 .. len) into acc (this lane's
// KG columns; ys points at the lane's first column of row 0 of the group, rows
// Sp elements apart): 32 ids per coalesced load, then kDepth rows in flight.
template <typename TY, int KG, typename A>
__device__ __forceinline__ void sum_rows(const Dev& d, const int* p, int len, const TY* ys, int Sp,
                                         A (&acc)[KG], int idx0, const L2Pol& pol, unsigned long long cold,
                                         int hot_n, bool on) {
  constexpr int D = ColGroup<TY, KG>::kDepth;
  const int lane = threadIdx.x & 31;
  for (int b = 0; b < len; b += 32) {
    const int cnt = min(32, len - b);
    // ids of the first block may come preloaded (idx0 >= 0 on every lane)
    const int idx = list_id(d, (b == 0 && __all_sync(0xffffffffu, idx0 >= 0)) ? idx0
                               : (lane < cnt ? __ldg(p + b + lane) : 0), b + lane);
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

__device__ __forceinline__ void bf16x4(uint2 x, float* f) {
  f[0] = __uint_as_float(x.x << 16);
  f[1] = __uint_as_float(x.x & 0xFFFF0000u);
  f[2] = __uint_as_float(x.y << 16);
  f[3] = __uint_as_float(x.y & 0xFFFF0000u);
}

__device__ __forceinline__ unsigned pack_bf16x2(float a, float b) {
  return (unsigned)__bfloat16_as_ushort(__float2bfloat16_rn(a)) |
         ((unsigned)__bfloat16_as_ushort(__float2bfloat16_rn(b)) << 16);
}

// (double)x for a nonzero x, exact up to 2^63 (step values are at most 2): scaled by 2^64,
// which makes subnormals normal, and put together in four integer operations. The
// conversion itself runs at the double rate, 16 cycles of the SM per warp.
__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double widen(float x) {
  const int b = __float_as_int(x * 0x1p64f);
  return __hiloint2double(((b >> 3) & 0x8FFFFFFF) + 0x34000000, b << 29);
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

// ---------------------------------------------------------------------------
// Tensor-core gather for bf16 rows of a group of G = 32 KG columns (64 KG
// bytes). Summing the gathered rows of each node is the product of the rows with
// a 0/1 matrix "edge belongs to node": for 16 edges and 8 nodes, mma.m16n8k16
//   A = rows transposed (m = columns, G / 16 tiles; k = edges),
//   B = membership      (k = edges, n = nodes, entries 1.0 or 0.0),
//   D = sums            (m = columns, n = nodes, float accumulation).
// Products with 1.0 and 0.0 are exact; the sums are float sums, truncated, and so kept
// to short chains (mma_put). A warp keeps a ring of kStages stages of 16 rows in shared
// memory: cp.async brings the rows in (16 bytes a lane, no registers held),
// ldmatrix.trans takes them out as A fragments, and a membership entry is one
// comparison of the edge's node number.
// Adding the rows in lanes took 13 warp instructions per edge and 32 columns
// (four conversions and two packed additions a row and lane, a node test, a
// flush per run); this form takes about 2. The kernel had been bound by
// instruction issue: with all memory traffic cut out it ran 25% faster only.
// tcgen05.mma reads both operands from shared memory and its sums from tensor
// memory; at 8 nodes a tile the membership operand alone would cost more stores
// than the rows, so the register-fed form is used.
// Rows of running columns are finite (|x| <= 2), so a zero entry never makes one
// NaN; whatever a stopped column holds stays in its own row of D, unused.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void cp_async16(unsigned smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Shared memory of one warp. Ring stages of kRs rows; 16 warps an SM
// (registers), with as many stages as 227 KB then leave room for.
template <typename TY, int KG>
struct RingWarp {
  static constexpr bool kMma = std::is_same<TY, __nv_bfloat16>::value;
  static constexpr int G = 32 * KG;
  static constexpr int kRow = G * (int)sizeof(TY);      // bytes of a row
  static constexpr int kChunks = kRow / 16;             // 16-byte chunks of a row
  static constexpr int kRs = kMma || kRow <= 256 ? 16 : 8;  // rows of a stage
  static constexpr int kStageBytes = kRs * kRow;        // 1 to 4 KB
  static constexpr int kStages = kMma ? (KG == 4 ? 2 : 4) : kStageBytes > 2048 ? 3 : 4;
  static constexpr int kWarps = 8;  // of a CTA
  static constexpr int kCtas = 2;   // per SM
  static_assert(kChunks <= 32 && kRow * kRs <= 4096, "a stage is one chunk a lane, up to eight times");
  alignas(128) unsigned char rows[kStages * kStageBytes];
  alignas(16) float acc[kMma ? 8 : 1][kMma ? G + 4 : 4];  // bf16: sums of eight nodes, by node and slot
  static constexpr bool kDouble = std::is_same<TY, double>::value;
  alignas(16) TY aside[kDouble ? G : 8];  // double: what was put aside of a long list's sum
  alignas(16) unsigned words[4][32];  // edges of four windows: row | node of the run << 25
  alignas(8) uint2 lists[32];       // nonempty lists of a run: pool offset - position, node << 25
};

// Byte offset of 16-byte chunk ch of row r in a stage, swizzled so that eight
// consecutive rows' chunks lie in different banks.
template <int KG>
__device__ __forceinline__ int row_chunk(int r, int ch) {
  const int sw = KG == 1 ? ch ^ ((r >> 1) & 3) : (ch & 8) | ((ch ^ r) & 7);
  return r * (64 * KG) + 16 * sw;
}

// 32-slot parts of a group up to its last running column (am: running slots).
template <int KG>
__device__ __forceinline__ int running_parts(const unsigned* am) {
  int p = 1;
#pragma unroll
  for (int k = 1; k < KG; ++k)
    if (am[k]) p = k + 1;
  return p;
}

// Copy the rows of words w[0 .. kRs) into a stage (chunks with a running column).
template <typename TY, int KG>
__device__ __forceinline__ void stage_rows(unsigned stage, const unsigned* w, const char* src,
                                           bool on) {
  using W = RingWarp<TY, KG>;
  constexpr int kPer = W::kRs * W::kChunks / 32;  // rows a lane copies its chunk of
  static_assert(kPer % 2 == 0, "row words are read in pairs");
  const int lane = threadIdx.x & 31;
  const int r0 = lane / W::kChunks * kPer, ch = lane % W::kChunks;
  if (on) {
    const char* from = src + 16 * ch;
#pragma unroll
    for (int i = 0; i < kPer; i += 2) {
      const uint2 u = *reinterpret_cast<const uint2*>(w + r0 + i);
      const int c0 = W::kMma ? row_chunk<KG>(r0 + i, ch) : (r0 + i) * W::kRow + 16 * ch;
      const int c1 = W::kMma ? row_chunk<KG>(r0 + i + 1, ch) : (r0 + i + 1) * W::kRow + 16 * ch;
      cp_async16(stage + c0, from + (size_t)(u.x & 0x1FFFFFFu) * W::kRow);
      cp_async16(stage + c1, from + (size_t)(u.y & 0x1FFFFFFu) * W::kRow);
    }
  }
}

// Does the chunk that this lane copies hold a running slot (am: running slots)?
template <typename TY, int KG>
__device__ __forceinline__ bool chunk_runs(const unsigned* am) {
  constexpr int per = 16 / (int)sizeof(TY);  // slots of a chunk
  const int q = (threadIdx.x & 31) % RingWarp<TY, KG>::kChunks * per;
  return ((am[q >> 5] >> (q & 31)) & ((1u << per) - 1u)) != 0;
}

// Membership of two edges in a node: two bf16 ones or zeros.
__device__ __forceinline__ unsigned member2(uint2 u, unsigned node) {
  return ((u.x >> 25) == node ? 0x3F80u : 0u) | ((u.y >> 25) == node ? 0x3F800000u : 0u);
}

// d += the 16 rows of a stage for membership (b0, b1). Tile f of d: d[4 f],
// d[4 f + 1] = slot 16 f + g of nodes 2 t, 2 t + 1; d[4 f + 2], d[4 f + 3] = slot
// 16 f + 8 + g. Only the first `parts` 32-slot parts are summed.
template <int KG>
__device__ __forceinline__ void mma_stage(float (&d)[8 * KG], unsigned stage, unsigned b0, unsigned b1,
                                          int parts) {
  const int lane = threadIdx.x & 31;
  const int r = (lane & 7) + 8 * (lane >> 4), c = (lane >> 3) & 1;
#pragma unroll
  for (int f = 0; f < 2 * KG; ++f) {
    if (f >= 2 * parts) break;  // warp-uniform: no column of the later parts runs
    unsigned a0, a1, a2, a3;
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(a0), "=r"(a1), "=r"(a2), "=r"(a3)
                 : "r"(stage + row_chunk<KG>(r, 2 * f + c))
                 : "memory");
    float* t = d + 4 * f;
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
        "{%8, %9}, {%0, %1, %2, %3};"
        : "+f"(t[0]), "+f"(t[1]), "+f"(t[2]), "+f"(t[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
  }
}

// A stream of E >= 1 edges, 32 a window, through the ring: word_at(w) gives lane
// = position of window w its word (any valid row for positions past the end, no
// node), eat(h, words, stage) consumes the kRs edges from h kRs on.
template <typename TY, int KG, typename WordF, typename EatF>
__device__ __forceinline__ void ring_stream(int E, RingWarp<TY, KG>& W, const char* src, bool on,
                                            WordF word_at, EatF eat) {
  using RW = RingWarp<TY, KG>;
  constexpr int S = RW::kStages, RS = RW::kRs, PW = 32 / RS;  // stages, rows a stage, stages a window
  static_assert((S - 1 + PW - 1) / PW + 1 <= 3, "four windows of words are kept");
  const int lane = threadIdx.x & 31;
  const int nh = (E + RS - 1) / RS, nwin = (E + 31) >> 5;
  const unsigned rows = smem_u32(W.rows);
  unsigned n0 = word_at(0), n1 = nwin > 1 ? word_at(1) : 0u;
  int slot = 0;  // ring slot of the stage issued next
  auto issue = [&](int s) {
    if (s < nh) {
      const int w = s / PW;
      if (s % PW == 0) {
        W.words[w & 3][lane] = n0;
        __syncwarp();
        n0 = n1;
        if (w + 2 < nwin) n1 = word_at(w + 2);
      }
      stage_rows<TY, KG>(rows + (unsigned)slot * RW::kStageBytes, W.words[w & 3] + RS * (s % PW), src, on);
      slot = slot + 1 == S ? 0 : slot + 1;
    }
    cp_async_commit();
  };
  __syncwarp();  // the last stream's words and rows have been read
#pragma unroll
  for (int s = 0; s < S - 1; ++s) issue(s);
  int from = 0;
  for (int h = 0; h < nh; ++h) {
    cp_async_wait<S - 2>();
    __syncwarp();  // stage h has landed for the whole warp, stage h - 1 has been read
    issue(h + S - 1);
    eat(h, W.words[(h / PW) & 3] + RS * (h % PW), rows + (unsigned)from * RW::kStageBytes);
    from = from + 1 == S ? 0 : from + 1;
  }
}

// The words of a piece of a long in-list (ids p[0 .. L), L >= 1): node 0.
__device__ __forceinline__ unsigned piece_word(const Dev& d, const int* p, int L, int w) {
  const int q = 32 * w + (threadIdx.x & 31);
  return (unsigned)list_id(d, __ldg(p + min(q, L - 1)), q) | (q < L ? 0u : 127u << 25);
}

// The in-lists of a run of up to 32 nodes as one edge stream: lane j holds node
// j's list length ll (0 to leave it out) and pool offset off. word() gives the
// windows' words, in order.
template <typename TY, int KG>
struct RunWords {
  const Dev& d;
  int P, E, started;  // first position of the lane's list, edges of the run, last list's rank
  int ll;
  __device__ __forceinline__ RunWords(const Dev& dev, int l, unsigned off, int incl, RingWarp<TY, KG>& W)
      : d(dev), P(incl - l), E(__shfl_sync(0xffffffffu, incl, 31)), started(-1), ll(l) {
    const int lane = threadIdx.x & 31;
    __syncwarp();  // the last run's list table has been read
    const unsigned full = __ballot_sync(0xffffffffu, ll > 0);
    if (ll > 0) W.lists[__popc(full & lanemask_lt())] = make_uint2(off - (unsigned)P, (unsigned)lane << 25);
    __syncwarp();
  }
  __device__ __forceinline__ unsigned word(int w, const RingWarp<TY, KG>& W) {
    const int lane = threadIdx.x & 31;
    const unsigned at = (unsigned)(P - 32 * w);
    const unsigned hm = __reduce_or_sync(0xffffffffu, ll > 0 && at < 32u ? 1u << at : 0u);
    const int q = 32 * w + lane;
    const uint2 l = W.lists[started + __popc(hm & (lanemask_lt() | (1u << lane)))];
    started += __popc(hm);
    // the sum wraps back; positions past the end repeat the last edge, for no node
    const int u = __ldg(d.pool_c + (l.x + (unsigned)min(q, E - 1)));
    return (unsigned)list_id(d, u, q) | (q < E ? l.y : 127u << 25);
  }
};

__device__ __forceinline__ int warp_inclusive(int x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// The tensor cores' float accumulator drops the bits that do not fit instead of rounding
// them, so a chain ends after kMmaChain stages of 16 rows: its sums are added, rounded to
// nearest, to those put aside in shared memory (`put`), each lane its own entries. Against
// the double sums of the same rows, lists of 1,000 came out 1.5 to 1.9 units of 2^-24 small
// on average, 0.03 to 0.05 so (0.35 in size; one lane addition after the other in pieces of
// 256, 0.3; with chains of 12 half a unit small); lists of 64 are exact either way. Only
// eight nodes with more than a chain's rows put anything aside: steps take 1 to 2% longer
// (131,071 nodes, 256 seeds 196 -> 201 us, 2^21 nodes 2,812 -> 2,841).
constexpr int kMmaChain = 8;
template <int KG>
__device__ __forceinline__ void mma_put(float (&d)[8 * KG], RingWarp<__nv_bfloat16, KG>& W, int parts,
                                        bool& put) {
  const int fg = (threadIdx.x & 31) >> 2, t2 = 2 * (threadIdx.x & 3);
#pragma unroll
  for (int f = 0; f < 4 * KG; ++f) {
    if (f >= 4 * parts) break;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      float* a = &W.acc[t2 + q][8 * f + fg];
      *a = put ? *a + d[2 * f + q] : d[2 * f + q];
      d[2 * f + q] = 0.f;
    }
  }
  put = true;
}
// d += the sums put aside.
template <int KG>
__device__ __forceinline__ void mma_take(float (&d)[8 * KG], const RingWarp<__nv_bfloat16, KG>& W, int parts,
                                         bool& put) {
  if (!put) return;  // warp-uniform
  const int fg = (threadIdx.x & 31) >> 2, t2 = 2 * (threadIdx.x & 3);
#pragma unroll
  for (int f = 0; f < 4 * KG; ++f) {
    if (f >= 4 * parts) break;
    d[2 * f] += W.acc[t2][8 * f + fg];
    d[2 * f + 1] += W.acc[t2 + 1][8 * f + fg];
  }
  put = false;
}

// bf16: sum of the rows of one piece of a long in-list: in the lanes with t = 0,
// d[4 f] and d[4 f + 2] hold slots 16 f + g and 16 f + 8 + g. Row r adds to node r mod 8,
// eight sums of an eighth of the rows, which need three bits less; they are added up at
// the end.
template <int KG>
__device__ __forceinline__ void mma_piece(const Dev& dev, const int* p, int L, const char* src, bool on,
                                          int parts, RingWarp<__nv_bfloat16, KG>& W, float (&d)[8 * KG]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t2 = 2 * (lane & 3);
  const unsigned mine = (t2 == g ? 0xFFFFu : 0u) | (t2 + 1 == g ? 0xFFFF0000u : 0u);
#pragma unroll
  for (int k = 0; k < 8 * KG; ++k) d[k] = 0.f;
  ring_stream<__nv_bfloat16, KG>(
      L, W, src, on, [&](int w) { return piece_word(dev, p, L, w); },
      [&](int, const unsigned* w, unsigned stage) {
        const uint2 u0 = *reinterpret_cast<const uint2*>(w + t2);
        const uint2 u1 = *reinterpret_cast<const uint2*>(w + 8 + t2);
        mma_stage<KG>(d, stage, member2(u0, 0u) & mine, member2(u1, 0u) & mine, parts);
      });
#pragma unroll
  for (int f = 0; f < 4 * KG; ++f) {
    if (f >= 4 * parts) break;  // warp-uniform
    float x = d[2 * f] + d[2 * f + 1];
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    x += __shfl_xor_sync(0xffffffffu, x, 2);
    d[2 * f] = x;
  }
}

// bf16: a run's lists. The nodes are taken eight at a time: finish(c, d) gets the
// sums of nodes 8 c .. 8 c + 7 (fragments as in mma_stage), in order, once each.
template <int KG, typename F>
__device__ __forceinline__ void mma_stream(const Dev& dev, int ll, unsigned off, const char* src,
                                           bool on, int parts, RingWarp<__nv_bfloat16, KG>& W, F finish) {
  const int lane = threadIdx.x & 31, t2 = 2 * (lane & 3);
  const int incl = warp_inclusive(ll);
  float d[8 * KG];
#pragma unroll
  for (int k = 0; k < 8 * KG; ++k) d[k] = 0.f;
  int c = 0;  // eight nodes being summed, and the stream position after them
  int Ec = __shfl_sync(0xffffffffu, incl, 7);
  int since = 0;     // stage from which those nodes' sums are in d
  bool put = false;  // what came before lies aside
  RunWords<__nv_bfloat16, KG> R(dev, ll, off, incl, W);
  if (R.E > 0) {
    ring_stream<__nv_bfloat16, KG>(
        R.E, W, src, on, [&](int w) { return R.word(w, W); },
        [&](int h, const unsigned* w, unsigned stage) {
          const uint2 u0 = *reinterpret_cast<const uint2*>(w + t2);
          const uint2 u1 = *reinterpret_cast<const uint2*>(w + 8 + t2);
          for (;;) {
            if (Ec > 16 * h) {
              const unsigned node = (unsigned)(8 * c + (lane >> 2));
              mma_stage<KG>(d, stage, member2(u0, node), member2(u1, node), parts);
            }
            if (Ec > 16 * h + 16) {  // goes on in the next half window
              if (h - since >= kMmaChain - 1) {
                mma_put<KG>(d, W, parts, put);
                since = h + 1;
              }
              break;
            }
            mma_take<KG>(d, W, parts, put);
            finish(c, d);
#pragma unroll
            for (int k = 0; k < 8 * KG; ++k) d[k] = 0.f;
            since = h;
            if (++c == 4) break;
            Ec = __shfl_sync(0xffffffffu, incl, 8 * c + 7);
          }
        });
  } else {
    for (; c < 4; ++c) finish(c, d);
  }
}

// ---------------------------------------------------------------------------
// float and double rows go through the same ring and are added by the lanes,
// lane l the slots [KG l, KG (l + 1)) of each row: one shared load and KG (float:
// KG / 2 packed) additions a row, a node's sum staying in registers from its
// first row to its last (NodeSum). A node's rows within a stage are summed by themselves
// (float: in two chains) and then added to the node's sum, which double rows and float
// rows of 128 columns put aside every kSumStages stages, so that the depth of their sum of
// k rows is kRs + kSumStages + k / (kRs kSumStages): one chain of 500 doubles was off by 3
// to 8 units of 2^-53, these sums by 0.7 (lane gathers 0.9), stages of 8 floats in one
// chain by 1.6 of 2^-24, so by 0.7 (lane gathers 0.95); stages of 16 floats (512 rows at
// most to a piece) by 1.2, bulk copies by 1.3. Double rows are bound by their additions,
// 16 cycles of the SM per row of 32 columns: a stage's first row starts its chain without
// one, which pays for the addition to the node's sum.
// ---------------------------------------------------------------------------
constexpr int kSumStages = 16;
template <int KG>
__device__ __forceinline__ void add_row(float (&a)[KG], const float (&x)[KG]) {
  if constexpr (KG == 1) {
    a[0] += x[0];
  } else {
#pragma unroll
    for (int k = 0; k < KG; k += 2) {
      unsigned long long u, v;
      asm("mov.b64 %0, {%1, %2};" : "=l"(u) : "f"(a[k]), "f"(a[k + 1]));
      asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(x[k]), "f"(x[k + 1]));
      asm("add.rn.f32x2 %0, %0, %1;" : "+l"(u) : "l"(v));
      asm("mov.b64 {%0, %1}, %2;" : "=f"(a[k]), "=f"(a[k + 1]) : "l"(u));
    }
  }
}
template <int KG>
__device__ __forceinline__ void add_row(double (&a)[KG], const double (&x)[KG]) {
#pragma unroll
  for (int k = 0; k < KG; ++k) a[k] += x[k];
}

// A node's sum: acc, and what was put aside of a long list: double rows in shared memory,
// each lane its own slots, if anything (`put`, warp-uniform); float rows of 128 columns
// (stages of 8) in registers; narrower float rows put nothing aside.
template <typename TY, int KG>
struct NodeSum {
  static constexpr bool kDouble = RingWarp<TY, KG>::kDouble;
  static constexpr bool kAside = kDouble || KG == 4;
  alignas(16) TY acc[KG];
  TY regs[kDouble ? 1 : KG];
  TY* mem;
  bool put;
  unsigned cur;  // the node being summed (127: none yet)
  __device__ __forceinline__ NodeSum(unsigned node, RingWarp<TY, KG>& W)
      : mem(W.aside + (kDouble ? (threadIdx.x & 31) * KG : 0)), cur(node) {
    clear();
  }
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int k = 0; k < KG; ++k) acc[k] = (TY)0;
    put = false;
    if constexpr (kAside && !kDouble) {
#pragma unroll
      for (int k = 0; k < KG; ++k) regs[k] = (TY)0;
    }
  }
  __device__ __forceinline__ void put_aside() {
    if constexpr (kDouble) {
      complete();
      store_k<TY, KG>(mem, acc);
      clear();
      put = true;
    } else if constexpr (kAside) {
      add_row<KG>(regs, acc);
#pragma unroll
      for (int k = 0; k < KG; ++k) acc[k] = (TY)0;
    }
  }
  __device__ __forceinline__ void complete() {
    if constexpr (kDouble) {
      if (put) {
        alignas(16) TY a[KG];
        load_k<TY, KG>(mem, a);
        add_row<KG>(acc, a);
      }
    } else if constexpr (kAside) {
      add_row<KG>(acc, regs);
    }
  }
};

// Rows of stage h, each added to its node's sum; done(node) is called after a node's last
// row, with the sum in S.acc (which then starts again from zero). kLong: the stream holds a
// list of more than kSumStages stages; without one nothing is put aside (double only; 64
// seeds at 65,537 nodes 182 us a step, 192 with the sums put aside in registers and always
// added. Float rows of 128 columns take one form: 256 columns of 2^18 nodes 509 us against
// 494 with one chain, 510 with two forms, 514 through shared memory).
template <typename TY, int KG, bool kLong, typename F>
__device__ __forceinline__ void add_stage(int h, const unsigned* w, const unsigned char* stage,
                                          NodeSum<TY, KG>& S, F done) {
  using RW = RingWarp<TY, KG>;
  constexpr int RS = RW::kRs;
  const int lane = threadIdx.x & 31;
  const unsigned node = w[lane & (RS - 1)] >> 25;
  const unsigned prev = __shfl_up_sync(0xffffffffu, node, 1);
  // bit r: row r begins another node than the row before it
  const unsigned heads = __ballot_sync(0xffffffffu, lane < RS && node != (lane ? prev : S.cur));
  // the lane's slots of every row first: between the rows' additions a node may
  // end, and each load would come after what that stores and be waited for (the
  // wait for shared memory was the largest stall)
  const TY* row = reinterpret_cast<const TY*>(stage) + lane * KG;
  alignas(16) TY x[RS][KG];
#pragma unroll
  for (int r = 0; r < RS; ++r) load_k<TY, KG>(row + r * RW::G, x[r]);
  constexpr int kChains = std::is_same<TY, float>::value ? 2 : 1;
  TY part[kChains][KG];
#pragma unroll
  for (int c = 0; c < kChains; ++c)
#pragma unroll
    for (int k = 0; k < KG; ++k) part[c][k] = (TY)0;
  auto gather = [&]() {  // the stage's chains into the node's sum
    if constexpr (kChains == 2) add_row<KG>(part[0], part[1]);
    add_row<KG>(S.acc, part[0]);
  };
#pragma unroll
  for (int r = 0; r < RS; ++r) {
    if ((heads >> r) & 1u) {  // warp-uniform
      if (r > 0) gather();
      if (S.cur != 127u) {
        if constexpr (kLong) S.complete();
        done(S.cur);
      }
      S.clear();
      S.cur = __shfl_sync(0xffffffffu, node, r);
#pragma unroll
      for (int c = 0; c < kChains; ++c)
#pragma unroll
        for (int k = 0; k < KG; ++k) part[c][k] = kChains == 2 ? (TY)0 : x[r][k];
    } else if (kChains == 1) {
      if (r == 0) {
#pragma unroll
        for (int k = 0; k < KG; ++k) part[0][k] = x[0][k];
      } else {
        add_row<KG>(part[0], x[r]);
      }
    }
    if constexpr (kChains == 2) add_row<KG>(part[r & 1], x[r]);
  }
  gather();
  if constexpr (kLong)
    if (h % kSumStages == kSumStages - 1) S.put_aside();
}

// ---------------------------------------------------------------------------
// Narrow steps (bf16 rows, packed groups): once the only running columns are
// group slots 0..W-1 (W = 4 or 8), a step gathers W-value rows (8 or 16
// bytes) from a compact [node][W] block, whose rows of the nodes with
// out-edges (ids first in the degree order) mostly stay in L2, instead of the
// rows of a whole group (64 to 256 bytes). Lane = position of the in-list
// stream of 32 nodes: each lane loads one row, a segmented warp scan per
// column sums each node's run, and the run's last lane adds it to the node's
// sums in shared memory; then lane = node finishes. A step reads the rows the
// step before it wrote, in that step's layout (the group layout, or a compact
// block of 8 or 4 columns: W only shrinks within a call).
// ---------------------------------------------------------------------------
template <int W>
struct Narrow {
  const __nv_bfloat16* src;  // gather rows of the previous step (row u at src + u stride)
  int stride;                // its row length: that of a group (group 0), 8 or 4
  __nv_bfloat16* dst;        // next compact rows ([node][W])
  __nv_bfloat16* e;          // residual rows (group 0 of the group layout, slots 0..W-1 used)
  int estride;               // ... and their length
  int col[W];                // columns of R held by slots 0..W-1
  unsigned act;              // bit c: column col[c] runs
};

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

// Node v's sums x: R += x (running columns), |x| into l1, next compact row and
// residual w = x s + e_old (when v has out-edges). The score reductions are marked
// evict-first as in the group steps (2^23 nodes, 4 of 256 columns running: 2,040 -> 1,780
// us a step, 8: 2,670 -> 2,190).
template <int W>
__device__ __forceinline__ void narrow_finish(const Narrow<W>& N, const Multi& M, int v,
                                              const float (&x)[W], float s, bool has_in,
                                              unsigned long long once, double (&l1)[W]) {
  if (has_in) {
#pragma unroll
    for (int c = 0; c < W; ++c)
      if ((N.act >> c) & 1u) {
        red_add_once(M.r + (size_t)v * M.Sp + N.col[c], (double)x[c], once);
        l1[c] += fabs((double)x[c]);
      }
  }
  if (s != 0.f) {
    __nv_bfloat16* ep = N.e + (size_t)v * N.estride;
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
__device__ __forceinline__ void narrow_stream(const Dev& d, const Narrow<W>& N, int ll, unsigned off,
                                              float* acc_s) {
  const int lane = threadIdx.x & 31;
  int incl = ll;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  const int P = incl - ll;
  const int E = __shfl_sync(0xffffffffu, incl, 31);
  // windows of 32 positions with their loads in flight together; of eight (rows of 4) or
  // six the last ones of a run often lie past its end (the same steps 1,750 -> 1,720 and
  // 2,155 -> 2,080 us)
  constexpr int R = 4;
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
      if (q < E)
        row[r].load(N.src + (size_t)list_id(d, __ldg(d.pool_c + oj + (unsigned)(q - Pj)), q) * N.stride);
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
                                            float* acc_s, double* my_part, Ctl* ctl,
                                            unsigned long long once) {
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
          if (e < Lp) rw[r].load(N.src + (size_t)list_id(d, __ldg(pl + e), e) * N.stride);
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
          narrow_finish<W>(N, M, v, x, scale_of<float>(d, v), true, once, l1n);
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
      narrow_stream<W>(d, N, mine ? len : 0, off, acc_s);
      __syncwarp();
      if (fin) {
        float x[W];
#pragma unroll
        for (int c = 0; c < W; ++c) x[c] = acc_s[lane * W + c];
        narrow_finish<W>(N, M, vl, x, sc, len > 0, once, l1n);
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

// Whole last CTA: per-column stopping from the step's column sums (added up by
// the CTAs' atomics: summing per-CTA partials here cost 456 double additions a
// column, 30 us a step of 256 columns at 16 cycles a warp), the call's stop, the column groups still running and
// the history entry (max over the columns that ran the step). A column whose
// x(0) is exactly zero has only zero terms: under the eps rule its one
// do-while step is counted and it stops at once.
// s_key (kMaxSeeds doubles) is shared-memory scratch of the caller (a buffer
// that is idle at the grid barrier).
template <int KG>
__device__ void decide_multi(const Dev& d, const PropParams& pp, int it, long long m,
                             double* s_key, bool narrow_rows) {
  constexpr int G = 32 * KG;
  const Multi& M = d.mu;
  const int Sp = M.Sp;
  Ctl* ctl = d.ctl;
  __shared__ double s_max[32];
  __shared__ unsigned s_gmask;
  __shared__ int s_maxslot;
  if (threadIdx.x == 0) {
    s_gmask = 0;
    s_maxslot = -1;
  }
  const bool pack = M.pack != 0;
  __syncthreads();
  double seen = 0.0;
  int live = 0;
  for (int j = threadIdx.x; j < Sp; j += blockDim.x) {
    double* tot = M.part + (it & 1) * Sp + j;
    const double L = __ldcg(tot);
    *tot = 0.0;
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
        // hold float sums of at most 32 nonnegative terms (bf16 rows; relative error
        // below 2^-19), hence the margin
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
    for (int i = 0; i < (int)blockDim.x / 32; ++i) mx = fmax(mx, s_max[i]);
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
    ctl->narrow = narrow_rows && M.yn0 != nullptr && ng == 1 && ctl->grp[0] == 0 && s_maxslot < 8
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
// consecutive columns (8 sectors) of the target's row. An item has three
// weights (kept, removed, new), so the products are formed once an item: one
// double multiplication per entry and 32 columns, at 16 cycles of the SM, and a
// walk entry by entry through the unchanged ones bound the kernel before (2^18
// nodes, 64 seeds, 1,000 edge ops: 258 -> 69 us; 131,071 nodes, 100 seeds: 152 ->
// 60 us). The binary searches run on the part of the other list that the item's
// first and last entry bound.
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
    unsigned nz = 0;  // bit k: some column of part k has a score
    unsigned mine = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) ru[k] = __ldcg(d.mu.r + (size_t)u * Sp + lane + 32 * k);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      nz |= (unsigned)__any_sync(0xffffffffu, ru[k] != 0.0) << k;
      mine |= (unsigned)(ru[k] != 0.0) << k;
    }
    if (!nz) continue;
    const double wa = L ? c1 / (double)L : 0.0;
    const double wb = dp ? c1 / (double)dp : 0.0;
    const int* oldl = d.pool_r + d.rec_old_off[c];
    const int* newl = d.pool_r + d.rec_fbase[c];
    const int e0 = q * kPiece, e1 = min(e0 + kPiece, L + dp);
    // the other list's part that can hold this item's entries (both ascend):
    // lanes 0 and 1 bound the old entries' part of the new list, 2 and 3 the new
    // entries' part of the old list
    int bound = 0;
    {
      const int o0 = min(e0, L), o1 = min(e1, L), n0 = max(e0 - L, 0), n1 = max(e1 - L, 0);
      if (lane == 0 && o0 < o1) bound = lower_bound_i(newl, dp, oldl[o0]);
      if (lane == 1 && o0 < o1) bound = lower_bound_i(newl, dp, oldl[o1 - 1] + 1);
      if (lane == 2 && n0 < n1) bound = lower_bound_i(oldl, L, newl[n0]);
      if (lane == 3 && n0 < n1) bound = lower_bound_i(oldl, L, newl[n1 - 1] + 1);
    }
    const int nb0 = __shfl_sync(0xffffffffu, bound, 0), nb1 = __shfl_sync(0xffffffffu, bound, 1);
    const int ob0 = __shfl_sync(0xffffffffu, bound, 2), ob1 = __shfl_sync(0xffffffffu, bound, 3);
    // one pass an entry kind: 0 kept, (1-c)(1/d' - 1/d), nothing when the degree
    // did not change; 1 removed; 2 new
    for (int eb = e0; eb < e1; eb += 32) {
      const int e = eb + lane;
      int a = 0, kind = 3;
      if (e < e1) {
        if (e < L) {
          a = oldl[e];
          kind = contains_i(newl + nb0, nb1 - nb0, a) ? 0 : 1;
        } else {
          a = newl[e - L];
          kind = contains_i(oldl + ob0, ob1 - ob0, a) ? 3 : 2;
        }
      }
      if (!OSP_GUARD(ctl, a >= 0 && a < d.nc, "multi offset target", c, e, a)) kind = 3;
      for (int t = 0; t < 3; ++t) {
        const double w = t == 0 ? wb - wa : t == 1 ? -wa : wb;
        unsigned m = __ballot_sync(0xffffffffu, kind == t);
        if (!m || w == 0.0) continue;  // warp-uniform
        double x[K];
#pragma unroll
        for (int k = 0; k < K; ++k) x[k] = (nz >> k) & 1u ? w * ru[k] : 0.0;
        hit |= mine;
        if ((m >> lane) & 1u) d.mark[a] = epoch;
        for (; m; m &= m - 1) {
          const int aj = __shfl_sync(0xffffffffu, a, __ffs(m) - 1);
          double* row = d.mu.xacc + (size_t)aj * Sp + lane;
#pragma unroll
          for (int k = 0; k < K; ++k)
            if ((mine >> k) & 1u) atomicAdd(row + 32 * k, x[k]);
        }
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

// CTAs per SM the generic seed-block kernel is built for: three when a lane's
// share of a gather row is at most 4 bytes (few registers), else two.
template <typename TY, int KG>
struct MultiOcc {
  static constexpr int value = KG * (int)sizeof(TY) <= 4 ? 3 : 2;
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
  __shared__ BarShared sh;
  __shared__ double s_part[kMaxSeeds];  // per column |x| sums of the CTA (shared-memory atomics)
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
  const size_t gs = (size_t)d.nc * G;  // gather block: elements per column group
  const int n = ctl->n;
  const long long m = ctl->m;
  const int epoch = ctl->epoch;
  const int n_pieces = ctl->n_pieces;
  const int n_tasks = ctl->n_tasks;
  const int hub_thr = ctl->hub_thr, hub_piece = ctl->hub_piece;
  const L2Pol pol = make_l2pol();
  const int hot_n = pp.hot_n;
  const unsigned long long cold = hot_n > 0 ? pol.once : pol.normal;
  TY* yb[2] = {(TY*)M.y0, (TY*)M.y1};
  TY* eb = (TY*)M.e;
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  double* my_part = s_part;
  if (blockIdx.x == 0 && threadIdx.x == 0) d.step_ns[0] = global_ns();

  // the CTA's column sums into the step's totals (by step parity; the decision
  // clears them for the step after next)
  auto column_sums = [&](int it) {
    __syncthreads();
    for (int j = threadIdx.x; j < Sp; j += blockDim.x) {
      const double a = s_part[j];
      if (a != 0.0) atomicAdd(M.part + (it & 1) * Sp + j, a);
    }
  };

  // x(0): stamped rows move from xacc into R and, scaled, into y(0); every
  // node with out-edges gets its y(0) row (zero when not stamped) in each
  // column group that has a nonzero offset entry
  {
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
    column_sums(0);
    if (bar_arrive(ctl, sh)) decide_multi<KG>(d, pp, 0, m, nullptr, false);
    if (!bar_release(ctl, sh)) return;
  }

  A* hub_acc = (A*)M.hub_acc;
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
    int cur = -1;  // column group of the items this warp works on now
    unsigned act = 0;
    double l1[KG];
#pragma unroll
    for (int k = 0; k < KG; ++k) l1[k] = 0.0;
    auto flush = [&]() {
      if (cur >= 0) {
#pragma unroll
        for (int k = 0; k < KG; ++k) {
          atomicAdd(my_part + cur * G + lane * KG + k, l1[k]);
          l1[k] = 0.0;
        }
      }
    };
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
#pragma unroll
        for (int k = 0; k < KG; ++k)
          act |= (unsigned)(*(volatile int*)&M.active[g * G + lane * KG + k] != 0) << k;
      }
      const TY* ysg = ys + g * gs;           // the group's gather rows, G elements apart
      const TY* ysl = ysg + lane * KG;       // this lane's columns of them
      const size_t c0 = (size_t)g * G + lane * KG;  // slot: gather rows, residuals, hub sums
      auto rbase_of = [&](int v) { return (size_t)v * Sp + c0; };
      auto ybase_of = [&](int v) { return g * gs + (size_t)v * G + lane * KG; };
      if (ti < n_pieces) {
        // a piece of a long in-list; the piece that completes the list finishes it
        const int h = __ldg(d.piece_hub + ti);
        const int v = __ldg(d.hubs + h);
        const int piece = ti - __ldg(d.hub_pstart + h);
        const int full = __ldg(d.len_c + v);
        const int* p = d.pool_c + __ldg(d.off_c + v) + (unsigned)(piece * hub_piece);
        const int L = min(hub_piece, full - piece * hub_piece);
        A acc[KG];
#pragma unroll
        for (int k = 0; k < KG; ++k) acc[k] = (A)0;
        if constexpr (kBulk) ring_sum_list<TY, KG, A>(rg, d, p, L, ysg, acc, pol, cold, hot_n);
        else sum_rows<TY, KG, A>(d, p, L, ysl, G, acc, -1, pol, cold, hot_n, act != 0);
        A* ha = hub_acc + (size_t)h * Sp + c0;
#pragma unroll
        for (int k = 0; k < KG; ++k) atomicAdd(ha + k, acc[k]);
        __threadfence();
        __syncwarp();  // every lane's additions come before lane 0's count
        int last = 0;
        if (lane == 0) {
          const int np = (full + hub_piece - 1) / hub_piece;
          last = atomicAdd(&M.hub_cnt[h * 8 + g], 1) == np - 1;
        }
        last = __shfl_sync(0xffffffffu, last, 0);
        if (last) {
          __threadfence();
          __syncwarp();  // ... and its count before every lane's reads
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
            sum_rows<TY, KG, A>(d, d.pool_c + off, len, ysl, G, acc, idx, pol, cold, hot_n, act != 0);
          finish_slice<TY, KG, A>(M, rbase_of(v), ybase_of(v), acc, s, len > 0, rr, eo, act, yd, l1, pol);
          if (!more) break;
        }
      }
    }
    flush();
    column_sums(it);
    if (bar_arrive(ctl, sh)) decide_multi<KG>(d, pp, it, m, nullptr, false);
    if (!bar_release(ctl, sh)) return;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) ctl->epoch = epoch + 1;
}


// The seed block through row rings (bf16 rows summed by the tensor cores, float
// and double rows by the lanes), one persistent cooperative launch per call.
// Columns are packed into groups of G = 32 KG slots: slot q holds column
// slot_col[q], chosen per call by the x(0) decision so that columns likely to
// run long share groups; R, the offsets and the per-column state stay by column,
// gather rows, residuals and partial sums by slot. A work item (a piece of a
// long in-list, or a task of consecutive nodes) is taken by one warp for all
// groups with a running column when there are several items a warp, so that its
// ids and headers come from L1 for the later groups; else for one group.
template <typename TY, int KG>
__global__ void __launch_bounds__(32 * RingWarp<TY, KG>::kWarps, RingWarp<TY, KG>::kCtas)
    k_propagate_ring(Dev d, PropParams pp) {
  using A = typename AccOf<TY>::type;
  using RW = RingWarp<TY, KG>;
  constexpr int G = 32 * KG;
  constexpr bool kMma = RW::kMma;
  __shared__ double s_part[kMaxSeeds];  // |x| of this step per column (shared-memory atomics)
  __shared__ double s_key[kMaxSeeds];
  __shared__ int s_col[kMaxSeeds];      // column of each slot
  __shared__ unsigned s_am[kMaxSeeds / 32];  // running slots
  __shared__ BarShared sh;
  __shared__ int s_grp[8];
  __shared__ int s_ngrp;
  extern __shared__ __align__(128) unsigned char dsm[];
  Ctl* ctl = d.ctl;
  if (*(volatile int*)&ctl->status) return;
  const Multi& M = d.mu;
  const int Sp = M.Sp;
  const size_t gs = (size_t)d.nc * G;  // gather block: elements per column group
  const int n = ctl->n;
  const long long m = ctl->m;
  const int epoch = ctl->epoch;
  const int n_pieces = ctl->n_pieces;
  const int n_tasks = ctl->n_tasks;
  const int hub_thr = ctl->hub_thr, hub_piece = ctl->hub_piece;
  const L2Pol pol = make_l2pol();
  TY* yb[2] = {(TY*)M.y0, (TY*)M.y1};
  __nv_bfloat16* eb = (__nv_bfloat16*)M.e;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  RW& W = reinterpret_cast<RW*>(dsm)[wid];
  double* my_part = s_part;
  for (int j = threadIdx.x; j < Sp; j += blockDim.x) s_part[j] = 0.0;
  __syncthreads();
  if (blockIdx.x == 0 && threadIdx.x == 0) d.step_ns[0] = global_ns();

  // the CTA's column sums into the step's totals (by step parity; the decision
  // clears them for the step after next)
  auto column_sums = [&](int it) {
    __syncthreads();
    for (int j = threadIdx.x; j < Sp; j += blockDim.x) {
      const double a = s_part[j];
      s_part[j] = 0.0;
      if (a != 0.0) atomicAdd(M.part + (it & 1) * Sp + j, a);
    }
  };

  // 1. ||x(0)||_1 per column from the stamped rows; the decision orders the
  //    columns by it (largest first: a larger offset needs more steps) into
  //    group slots and picks the groups that hold a running column
  unsigned tb = 0;  // bit k: column lane + 32 k has an offset entry
  for (int k = 0; k < 8 && lane + 32 * k < M.S; ++k)
    if (*(volatile int*)&M.touched[lane + 32 * k]) tb |= 1u << k;
  __syncthreads();
  double l0[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) l0[k] = 0.0;
  for (int vb = gw * 32; vb < n && __any_sync(0xffffffffu, tb != 0); vb += nw * 32) {
    const int vl = vb + lane;
    unsigned stamped = __ballot_sync(0xffffffffu, vl < n && __ldcg(d.mark + vl) == epoch);
    for (; stamped; stamped &= stamped - 1) {
      const int v = vb + __ffs(stamped) - 1;
      double x[8];
#pragma unroll
      for (int k = 0; k < 8; ++k)
        x[k] = (tb >> k) & 1u ? __ldcg(M.xacc + (size_t)v * Sp + lane + 32 * k) : 0.0;
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if ((tb >> k) & 1u) l0[k] += fabs(x[k]);
    }
  }
#pragma unroll
  for (int k = 0; k < 8; ++k)
    if ((tb >> k) & 1u) atomicAdd(my_part + lane + 32 * k, l0[k]);
  column_sums(0);
  if (bar_arrive(ctl, sh)) decide_multi<KG>(d, pp, 0, m, s_key, kMma);
  if (!bar_release(ctl, sh)) return;
  // 2. R += x(0) and the y(0) rows, in group slots
  if (threadIdx.x < 8) s_grp[threadIdx.x] = *(volatile int*)&ctl->grp[threadIdx.x];
  if (threadIdx.x == 0) s_ngrp = *(volatile int*)&ctl->n_grp;
  __syncthreads();
  const int ng = s_ngrp;
  // a lane's slots are lane, lane + 32, ...: 32-slot parts q of the groups
  int colq[8];
  unsigned actq = 0;  // bit q: this lane's column of part q runs
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    colq[q] = 0;
    if (32 * q < Sp) {
      colq[q] = __ldcg(M.slot_col + 32 * q + lane);
      if (*(volatile int*)&M.active[colq[q]]) actq |= 1u << q;
    }
  }
  for (int vb = gw * 32; vb < n && ng > 0; vb += nw * 32) {
    const int vl = vb + lane;
    const unsigned stamped = __ballot_sync(0xffffffffu, vl < n && __ldcg(d.mark + vl) == epoch);
    const A s_l = vl < n ? scale_of<A>(d, vl) : (A)0;
    // rows of nodes without an offset entry start at zero: 16 bytes a lane
    const unsigned blank = __ballot_sync(0xffffffffu, s_l != (A)0) & ~stamped;
    constexpr int kLanes = RW::kChunks;  // lanes a row
    for (int gi = 0; gi < ng && blank; ++gi) {
      const size_t at = s_grp[gi] * gs + (size_t)vb * G + 16 / sizeof(TY) * (lane % kLanes);
#pragma unroll
      for (int r = 0; r < kLanes; ++r) {
        const int j = r * (32 / kLanes) + lane / kLanes;
        if ((blank >> j) & 1u) {
          *reinterpret_cast<uint4*>(yb[0] + at + (size_t)j * G) = make_uint4(0u, 0u, 0u, 0u);
          if constexpr (kMma)
            *reinterpret_cast<uint4*>(eb + at + (size_t)j * G) = make_uint4(0u, 0u, 0u, 0u);
        }
      }
    }
    for (unsigned work = stamped; work; work &= work - 1) {
      const int jj = __ffs(work) - 1;
      const int v = vb + jj;
      const A s = __shfl_sync(0xffffffffu, s_l, jj);
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (!((actq >> q) & 1u)) continue;
        const size_t ybase = (q / KG) * gs + (size_t)v * G + 32 * (q % KG) + lane;
        TY yv = from_acc((A)0, (TY*)nullptr), ev = yv;
        const size_t rb = (size_t)v * Sp + colq[q];
        const double x = __ldcg(M.xacc + rb);
        if (x != 0.0) {
          M.r[rb] += x;
          M.xacc[rb] = 0.0;
          const A w = (A)x * s;
          yv = from_acc(w, (TY*)nullptr);
          if constexpr (kMma) ev = __float2bfloat16_rn(w - __bfloat162float(yv));
        }
        if (s != (A)0) {
          const TY y1[1] = {yv}, e1[1] = {ev};
          st_pol(yb[0] + ybase, y1, pol.once);
          if constexpr (kMma) st_pol(eb + ybase, e1, pol.once);
        }
      }
    }
  }
  if (bar_arrive(ctl, sh) && threadIdx.x == 0) ctl->ctr[1] = 0;
  if (!bar_release(ctl, sh)) return;

  A* hub_acc = (A*)M.hub_acc;
  int prev_narrow = 0;  // row width of the compact block the last step wrote (0: none)
  for (int it = 1;; ++it) {
    if (*(volatile int*)&ctl->stop) break;
    if (threadIdx.x < 8) s_grp[threadIdx.x] = *(volatile int*)&ctl->grp[threadIdx.x];
    if (threadIdx.x == 0) s_ngrp = *(volatile int*)&ctl->n_grp;
    for (int q = threadIdx.x; q < Sp; q += blockDim.x) {  // warps whole: Sp is a multiple of 32
      const int col = __ldcg(M.slot_col + q);
      const unsigned a = __ballot_sync(0xffffffffu, *(volatile int*)&M.active[col] != 0);
      s_col[q] = col;
      if (lane == 0) s_am[q >> 5] = a;
    }
    __syncthreads();
    const TY* ys = yb[(it - 1) & 1];
    TY* yd = yb[it & 1];
    const int n_items = n_pieces + n_tasks;
    const int narrow = kMma ? *(volatile int*)&ctl->narrow : 0;  // row width of a narrow step (0: over groups)
    if constexpr (kMma) {
      if (narrow) {
        __nv_bfloat16* yn[2] = {(__nv_bfloat16*)M.yn0, (__nv_bfloat16*)M.yn1};
        const __nv_bfloat16* src =
            prev_narrow ? yn[(it - 1) & 1] : ys;
        const int stride = prev_narrow ? prev_narrow : G;
        float* acc_s = &W.acc[0][0];
        static_assert(sizeof(W.acc) >= 256 * sizeof(float), "sums of a narrow run");
        if (narrow == 4) {
          Narrow<4> N{src, stride, yn[it & 1], eb, G, {}, 0u};
  #pragma unroll
          for (int c = 0; c < 4; ++c) {
            N.col[c] = __ldcg(M.slot_col + c);
            if (*(volatile int*)&M.active[N.col[c]]) N.act |= 1u << c;
          }
          narrow_step<4>(d, M, N, n_items, n_pieces, hub_thr, hub_piece, hub_acc, acc_s,
                         my_part, ctl, pol.once);
        } else {
          Narrow<8> N{src, stride, yn[it & 1], eb, G, {}, 0u};
  #pragma unroll
          for (int c = 0; c < 8; ++c) {
            N.col[c] = __ldcg(M.slot_col + c);
            if (*(volatile int*)&M.active[N.col[c]]) N.act |= 1u << c;
          }
          narrow_step<8>(d, M, N, n_items, n_pieces, hub_thr, hub_piece, hub_acc, acc_s,
                         my_part, ctl, pol.once);
        }
      }
    }
    prev_narrow = narrow;
    const int ng = s_ngrp;
    const bool whole = n_items >= 4 * nw;  // an item's groups by one warp
    const int total = narrow ? 0 : whole ? n_items : n_items * ng;
    for (int k = 0;; ++k) {
      int t = gw;  // the first item is the warp's own number, later ones come from the counter
      if (k > 0) {
        if (total <= nw) break;
        if (lane == 0) t = nw + atomicAdd(&ctl->ctr[1], 1);
        t = __shfl_sync(0xffffffffu, t, 0);
      }
      if (t >= total) break;
      const int ti = whole ? t : t / ng;
      const int g0 = whole ? 0 : t - ti * ng, g1 = whole ? ng : g0 + 1;
      if (ti < n_pieces) {
        // a piece of a long in-list; the piece that completes the list finishes it
        const int h = __ldg(d.piece_hub + ti);
        const int v = __ldg(d.hubs + h);
        const int piece = ti - __ldg(d.hub_pstart + h);
        const int full = __ldg(d.len_c + v);
        const int* p = d.pool_c + __ldg(d.off_c + v) + (unsigned)(piece * hub_piece);
        const int L = min(hub_piece, full - piece * hub_piece);
        const int np = (full + hub_piece - 1) / hub_piece;
        for (int gi = g0; gi < g1; ++gi) {
          const int g = s_grp[gi];
          const unsigned* am = s_am + g * KG;
          const bool on = chunk_runs<TY, KG>(am);
          const char* src = reinterpret_cast<const char*>(ys + g * gs);
          A* ha = hub_acc + (size_t)h * Sp + g * G;
          if constexpr (kMma) {
            float D[8 * KG];
            mma_piece<KG>(d, p, L, src, on, running_parts<KG>(am), W, D);
            if ((lane & 3) == 0) {
              const int fg = lane >> 2;
#pragma unroll
              for (int f = 0; f < 4 * KG; ++f)
                if ((am[f >> 2] >> (8 * (f & 3) + fg)) & 1u) atomicAdd(ha + 8 * f + fg, D[2 * f]);
            }
          } else {
            NodeSum<A, KG> sum(0u, W);
            auto add = [&](unsigned) {
#pragma unroll
              for (int k = 0; k < KG; ++k) atomicAdd(ha + lane * KG + k, sum.acc[k]);
            };
            ring_stream<TY, KG>(
                L, W, src, on, [&](int w) { return piece_word(d, p, L, w); },
                [&](int h, const unsigned* w, unsigned stage) {
                  // rows past the end begin "no node": the piece's sum is complete there
                  add_stage<TY, KG, true>(h, w, W.rows + (stage - smem_u32(W.rows)), sum, add);
                });
            if (sum.cur == 0u) {
              sum.complete();
              add(0u);
            }
          }
          __threadfence();
          __syncwarp();  // every lane's additions come before lane 0's count
          int last = 0;
          if (lane == 0) last = atomicAdd(&M.hub_cnt[h * 8 + g], 1) == np - 1;
          last = __shfl_sync(0xffffffffu, last, 0);
          if (last) {
            __threadfence();
            __syncwarp();  // ... and its count before every lane's reads
            if (lane == 0) M.hub_cnt[h * 8 + g] = 0;
            const A sv = scale_of<A>(d, v);
#pragma unroll
            for (int k = 0; k < KG; ++k) {  // lane = slot
              const A x = __ldcg(ha + 32 * k + lane);
              ha[32 * k + lane] = (A)0;
              if (!((am[k] >> lane) & 1u)) continue;
              const int col = s_col[g * G + 32 * k + lane];
              red_add_once(M.r + (size_t)v * Sp + col, (double)x, pol.once);
              atomicAdd(my_part + col, fabs((double)x));
              if (sv != (A)0) {
                const size_t at = g * gs + (size_t)v * G + 32 * k + lane;
                if constexpr (kMma) {
                  const float w = x * sv + __bfloat162float(eb[at]);
                  const __nv_bfloat16 yv = __float2bfloat16_rn(w);
                  yd[at] = yv;
                  eb[at] = __float2bfloat16_rn(w - __bfloat162float(yv));
                } else {
                  yd[at] = x * sv;
                }
              }
            }
          }
        }
        continue;
      }
      const int task = ti - n_pieces;
      const int c0t = __ldg(d.task_first + task), c1t = __ldg(d.task_first + task + 1);
      for (int gi = g0; gi < g1; ++gi) {
        const int g = s_grp[gi];
        const unsigned* am = s_am + g * KG;
        const int* scol = s_col + g * G;
        const char* src = reinterpret_cast<const char*>(ys + g * gs);
        const bool on = chunk_runs<TY, KG>(am);
        const int parts = running_parts<KG>(am);
        // float and double rows: this lane's slots lane KG + k, their columns
        int col[KG];
        unsigned amk = 0;
#pragma unroll
        for (int k = 0; k < KG; ++k) {
          const int q = lane * KG + k;
          col[k] = scol[q];
          amk |= ((am[q >> 5] >> (q & 31)) & 1u) << k;
        }
        // list lengths, offsets and scales of the next run of 32 nodes load
        // while the current run is summed
        int nx_len = 0;
        unsigned nx_off = 0;
        A nx_s = (A)0;
        auto header = [&](int vb) {
          const int vl = vb + lane;
          nx_len = 0;
          nx_off = 0;
          nx_s = (A)0;
          if (vl < c1t) {
            nx_len = __ldg(d.len_c + vl);
            nx_off = __ldg(d.off_c + vl);
            nx_s = scale_of<A>(d, vl);
          }
        };
        header(c0t);
        for (int vb = c0t; vb < c1t; vb += 32) {
          const int my_len = nx_len;
          const unsigned my_off = nx_off;
          const A my_s = nx_s;
          if (vb + 32 < c1t) header(vb + 32);
          const bool mine = vb + lane < c1t && my_len <= hub_thr;  // hubs go by pieces
          const unsigned fin = __ballot_sync(0xffffffffu, mine && (my_len > 0 || my_s != (A)0));
          if (!fin) continue;
          // |x| of the run, added to the FP64 partial once: in double, for bf16 rows in
          // float (at most 32 nonnegative terms)
          using L = std::conditional_t<kMma, float, double>;
          L l1f[KG];
#pragma unroll
          for (int k = 0; k < KG; ++k) l1f[k] = (L)0;
          if constexpr (kMma) {
            mma_stream<KG>(
                d, mine ? my_len : 0, my_off, src, on, parts, W, [&](int c, const float (&D)[8 * KG]) {
                  if (!((fin >> (8 * c)) & 0xFFu)) return;  // warp-uniform
                  // the sums by node and slot (conflict-free: banks 8 t + g)
                  const int fg = lane >> 2, t2 = 2 * (lane & 3);
  #pragma unroll
                  for (int f = 0; f < 4 * KG; ++f) {
                    if (f >= 4 * parts) break;
                    W.acc[t2][8 * f + fg] = D[2 * f];
                    W.acc[t2 + 1][8 * f + fg] = D[2 * f + 1];
                  }
                  // next gather row and residual: lane = node, every fourth
                  // chunk of four slots; the old residuals load first
                  const int j = lane >> 2, q = lane & 3;
                  const float sj = __shfl_sync(0xffffffffu, my_s, 8 * c + j);
                  const bool src_node = sj != 0.f && ((fin >> (8 * c + j)) & 1u);
                  const size_t at = g * gs + (size_t)(vb + 8 * c + j) * G + 4 * q;
                  uint2 eo[2 * KG];
  #pragma unroll
                  for (int i = 0; i < 2 * KG; ++i)
                    eo[i] = src_node && ((am[i >> 1] >> (16 * (i & 1) + 4 * q)) & 0xFu)
                                ? __ldcg(reinterpret_cast<const uint2*>(eb + at + 16 * i))
                                : make_uint2(0u, 0u);
                  __syncwarp();
                  // R += x: lane = slot (a node without in-list has x = 0)
                  double* rp = M.r + (size_t)(vb + 8 * c) * Sp;
  #pragma unroll
                  for (int k = 0; k < KG; ++k) {
                    if (k >= parts) break;
                    const bool run = (am[k] >> lane) & 1u;
                    double* rk = rp + scol[32 * k + lane];
  #pragma unroll
                    for (int jj = 0; jj < 8; ++jj) {
                      const float x = W.acc[jj][32 * k + lane];
                      if (run && x != 0.f) {
                        red_add_once(rk, widen(x), pol.once);
                        l1f[k] += fabsf(x);
                      }
                      rk += Sp;
                    }
                  }
  #pragma unroll
                  for (int i = 0; i < 2 * KG; ++i) {
                    if (i >= 2 * parts) break;
                    if (!(src_node && ((am[i >> 1] >> (16 * (i & 1) + 4 * q)) & 0xFu))) continue;
                    const float4 x = *reinterpret_cast<const float4*>(&W.acc[j][16 * i + 4 * q]);
                    const float w0 = x.x * sj + __uint_as_float(eo[i].x << 16);
                    const float w1 = x.y * sj + __uint_as_float(eo[i].x & 0xFFFF0000u);
                    const float w2 = x.z * sj + __uint_as_float(eo[i].y << 16);
                    const float w3 = x.w * sj + __uint_as_float(eo[i].y & 0xFFFF0000u);
                    const uint2 y = make_uint2(pack_bf16x2(w0, w1), pack_bf16x2(w2, w3));
                    *reinterpret_cast<uint2*>(yd + at + 16 * i) = y;
                    *reinterpret_cast<uint2*>(eb + at + 16 * i) =
                        make_uint2(pack_bf16x2(w0 - __uint_as_float(y.x << 16),
                                               w1 - __uint_as_float(y.x & 0xFFFF0000u)),
                                   pack_bf16x2(w2 - __uint_as_float(y.y << 16),
                                               w3 - __uint_as_float(y.y & 0xFFFF0000u)));
                  }
                  __syncwarp();  // acc is free again
                });
#pragma unroll
            for (int k = 0; k < KG; ++k)
              if (l1f[k] != 0.f) atomicAdd(my_part + scol[32 * k + lane], (double)l1f[k]);
          } else {
            // a node's next gather row; one without in-list writes zeros
            for (unsigned z = fin & __ballot_sync(0xffffffffu, my_len == 0); z; z &= z - 1) {
              alignas(16) const TY zero[KG] = {};
              store_k<TY, KG>(yd + g * gs + (size_t)(vb + __ffs(z) - 1) * G + lane * KG, zero);
            }
            const int ll = mine ? my_len : 0;
            RunWords<TY, KG> R(d, ll, my_off, warp_inclusive(ll), W);
            if (R.E == 0) continue;
            NodeSum<A, KG> sum(127u, W);
            const A(&acc)[KG] = sum.acc;
            auto done = [&](unsigned j) {  // node vb + j: x = acc
              const A sj = __shfl_sync(0xffffffffu, my_s, (int)j);
              double* rp = M.r + (size_t)(vb + j) * Sp;
#pragma unroll
              for (int k = 0; k < KG; ++k)
                if (((amk >> k) & 1u) && acc[k] != (A)0) {
                  const double x = widen(acc[k]);
                  red_add_once(rp + col[k], x, pol.once);
                  l1f[k] += fabs(x);
                }
              if (sj != (A)0) {
                alignas(16) TY yv[KG];
#pragma unroll
                for (int k = 0; k < KG; ++k) yv[k] = acc[k] * sj;
                store_k<TY, KG>(yd + g * gs + (size_t)(vb + j) * G + lane * KG, yv);
              }
            };
            auto stream = [&](auto longs) {
              ring_stream<TY, KG>(
                  R.E, W, src, on, [&](int w) { return R.word(w, W); },
                  [&](int h, const unsigned* w, unsigned stage) {
                    add_stage<TY, KG, decltype(longs)::value>(h, w, W.rows + (stage - smem_u32(W.rows)),
                                                              sum, done);
                  });
            };
            if constexpr (std::is_same<TY, float>::value) {
              stream(std::true_type{});
            } else {
              if (__reduce_max_sync(0xffffffffu, ll) > RW::kRs * kSumStages) stream(std::true_type{});
              else stream(std::false_type{});
            }
            if (sum.cur != 127u) {
              sum.complete();
              done(sum.cur);
            }
#pragma unroll
            for (int k = 0; k < KG; ++k)
              if (l1f[k] != 0.0) atomicAdd(my_part + col[k], l1f[k]);
          }
        }
      }
    }
    column_sums(it);
    if (bar_arrive(ctl, sh)) decide_multi<KG>(d, pp, it, m, s_key, kMma);
    if (!bar_release(ctl, sh)) return;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) ctl->epoch = epoch + 1;
}

namespace {

struct MultiFn {
  const void* fn;
  int smem;  // dynamic shared memory bytes
  int threads = kPropThreads;
};

template <typename TY, int KG>
MultiFn multi_fn_k(SeedRows rows) {
  if (rows == SeedRows::kBulk) return {(const void*)k_propagate_multi<TY, KG, true>, RingCfg<TY, KG>::kSmem};
  if constexpr (seed_ring_fits((int)sizeof(TY), KG))
    if (rows == SeedRows::kRing)
      return {(const void*)k_propagate_ring<TY, KG>,
              RingWarp<TY, KG>::kWarps * (int)sizeof(RingWarp<TY, KG>), 32 * RingWarp<TY, KG>::kWarps};
  return {(const void*)k_propagate_multi<TY, KG, false>, 0};
}

template <typename TY>
MultiFn multi_fn(int KG, SeedRows rows) {
  switch (KG) {
    case 1: return multi_fn_k<TY, 1>(rows);
    case 2: return multi_fn_k<TY, 2>(rows);
    case 4: return multi_fn_k<TY, 4>(rows);
    default: return multi_fn_k<TY, 8>(rows);
  }
}

MultiFn pick_multi(int precision, int KG, SeedRows rows) {
  if (precision == OSP_PREC_FP64) return multi_fn<double>(KG, rows);
  if (precision == OSP_PREC_FP32_ACC64) return multi_fn<float>(KG, rows);
  return multi_fn<__nv_bfloat16>(KG, rows);
}

}  // namespace

int propagate_multi_grid(int precision, int KG, int num_sms, SeedRows rows) {
  const MultiFn f = pick_multi(precision, KG, rows);
  if (f.smem > 0 &&
      cudaFuncSetAttribute(f.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, f.smem) != cudaSuccess)
    return 0;
  int bps = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, f.fn, f.threads, f.smem) != cudaSuccess ||
      bps <= 0)
    return 0;
  bps = bps > 4 ? 4 : bps;
  const int g = bps * num_sms;
  return g > kMaxGrid ? kMaxGrid : g;
}

cudaError_t launch_propagate_multi(const Dev& d, const PropParams& pp, int precision, int KG,
                                   int grid, SeedRows rows, cudaStream_t s) {
  Dev dd = d;
  PropParams p = pp;
  void* args[] = {&dd, &p};
  const MultiFn f = pick_multi(precision, KG, rows);
  return cudaLaunchCooperativeKernel(f.fn, dim3(grid), dim3(f.threads), args, (size_t)f.smem, s);
}

// ---------------------------------------------------------------------------
// Failure-detection self-tests: the bounded waits of the persistent kernels
// are made to run out on purpose (a CTA that never arrives; an mbarrier whose
// announced bytes never all land), and the status word must report it.
// ---------------------------------------------------------------------------
// Both grid barriers one after the other: the seed block's on ctl[0], the one-seed
// kernel's on ctl[1] (its arrivals in bar_count).
__global__ void k_selftest_barrier(Ctl* ctl, int lose) {
  __shared__ BarShared sh;
  if (lose && blockIdx.x == 0) return;  // this CTA never arrives
  if (bar_arrive(ctl, sh) && threadIdx.x == 0) ctl->iter = 1;
  bar_release(ctl, sh);
  if (threadIdx.x == 0 && grid_wait(&ctl[1].bar_count, gridDim.x, ctl + 1)) ctl[1].iter = 1;
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
