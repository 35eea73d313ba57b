// Sweep kernels: a program's expressions evaluated in one pass over its
// outputs (hiccl_sweep.cpp builds the classes; see there for why this equals
// the factorized schedule).
//
// What bounds a pass is memory: every input is read once and every output
// written once, with at most one add per value between.  A warp takes one
// unit -- V vectors of 32 lanes of one member -- and loads up to eight
// sources before it folds the first, so that 16 warps an SM hold 64 to 128
// KiB in flight; the value goes to every destination straight from
// registers.  CTAs are small (64 threads for folds), so that a finished warp's
// registers are not held by its slower neighbours: 635 against 641 us for the
// All-reduce below at 256 threads, 557 against 572 us for a group of 48
// collectives.  Nothing waits on another CTA, so the grid is one warp per unit
// and the hardware's CTA scheduler balances the tail: measured against a
// persistent grid of the same code, 41.3 against 74 us for a 4 MiB Broadcast
// to 64 ranks, 624 against 676 us for the All-reduce below; bulk (TMA) loads
// and stores through shared-memory rings measured 48.9 and 672 us.
//
// Against the step executor, GB300, a start as a program times it: All-reduce
// of 64 MiB a rank over 32 ranks 769 -> 646 us (626 us, 6.87 TB/s of the
// inputs read and outputs written once, without the host), All-reduce of 64
// KiB of BF16 over 8 ranks (graph replay) 22.6 -> 6.8 us, the seven
// collectives of 64 ranks x 4 MiB (graph replay) 456 -> 306 us, an odd-length
// 6 MiB All-reduce over 16 ranks 531 -> 54 us.

#include <cuda_runtime.h>

#include <type_traits>

#include "hiccl_device.cuh"
#include "hiccl_internal.h"
#include "hiccl_sweep.h"

namespace hiccl {

namespace {

// ---- accesses of W bytes per lane ----------------------------------------------

template <int W>
struct Raw {
  uint32_t w[W >= 4 ? W / 4 : 1];
};
// (L2 only: under programmatic launch another kernel may just have written
// these lines, and no input is read twice)
template <int W>
__device__ __forceinline__ Raw<W> ld_raw(unsigned long long a) {
  Raw<W> r;
  if constexpr (W == 16) {
    const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(a));
    r.w[0] = v.x;
    r.w[1] = v.y;
    r.w[2] = v.z;
    r.w[3] = v.w;
  } else if constexpr (W == 4) {
    r.w[0] = __ldcg(reinterpret_cast<const unsigned int *>(a));
  } else {
    r.w[0] = __ldcg(reinterpret_cast<const unsigned short *>(a));
  }
  return r;
}
template <int W>
__device__ __forceinline__ void st_raw(unsigned long long a, const Raw<W> &r) {
  if constexpr (W == 16) *reinterpret_cast<uint4 *>(a) = make_uint4(r.w[0], r.w[1], r.w[2], r.w[3]);
  else if constexpr (W == 4) *reinterpret_cast<unsigned int *>(a) = r.w[0];
  else *reinterpret_cast<unsigned short *>(a) = (unsigned short)r.w[0];
}

// ---- payload families -----------------------------------------------------------
// N 32-bit accumulators hold the W bytes of a lane: the words themselves
// (F32, I32), or BF16 values widened to binary32.

enum Family { F32_SUM, ANY_32, BF16_SUM, BF16_ANY };

template <int FAM, int W>
struct Acc {
  static constexpr bool BF = FAM == BF16_SUM || FAM == BF16_ANY;
  static constexpr int N = BF ? W / 2 : W / 4;

  __device__ __forceinline__ static uint32_t widen(const Raw<W> &r, int i) {
    if constexpr (!BF) return r.w[i];
    else return i & 1 ? r.w[i / 2] & 0xffff0000u : r.w[i / 2] << 16;
  }
  __device__ __forceinline__ static Raw<W> pack(const uint32_t *a) {
    Raw<W> r;
    if constexpr (!BF) {
#pragma unroll
      for (int i = 0; i < N; ++i) r.w[i] = a[i];
    } else if constexpr (W >= 4) {
#pragma unroll
      for (int i = 0; i < N / 2; ++i) r.w[i] = f32x2_to_bf16x2(__uint_as_float(a[2 * i]), __uint_as_float(a[2 * i + 1]));
    } else {
      r.w[0] = f32_to_bf16_rn(__uint_as_float(a[0]));
    }
    return r;
  }
  __device__ __forceinline__ static void round(uint32_t *a) {
    if constexpr (BF) {
      const Raw<W> r = pack(a);
#pragma unroll
      for (int i = 0; i < N; ++i) a[i] = widen(r, i);
    }
  }
};

// a[i] = a[i] op b(i) over n words, the operator's branch taken once (once per
// word, a 64-way int32 maximum of 1 MiB a rank took 39 us instead of 26)
template <int FAM, int N, typename F>
__device__ __forceinline__ void combine(uint32_t *a, F b, uint32_t dt, uint32_t rop) {
  auto f = [](uint32_t x) { return __uint_as_float(x); };
  auto each = [&](auto op) {
#pragma unroll
    for (int i = 0; i < N; ++i) a[i] = op(a[i], b(i));
  };
  auto add = [&](uint32_t x, uint32_t y) { return __float_as_uint(__fadd_rn(f(x), f(y))); };
  auto fmx = [&](uint32_t x, uint32_t y) { return __float_as_uint(fmaxf(f(x), f(y))); };
  auto fmn = [&](uint32_t x, uint32_t y) { return __float_as_uint(fminf(f(x), f(y))); };
  if constexpr (FAM == F32_SUM || FAM == BF16_SUM) {
    each(add);
  } else if constexpr (FAM == BF16_ANY) {
    if (rop == HICCL_MAX) each(fmx);
    else each(fmn);
  } else if (dt == HICCL_F32) {
    if (rop == HICCL_MAX) each(fmx);
    else each(fmn);
  } else {
    switch (rop) {
      case HICCL_SUM: each([](uint32_t x, uint32_t y) { return x + y; }); break;
      case HICCL_MAX: each([](uint32_t x, uint32_t y) { return (uint32_t)max((int)x, (int)y); }); break;
      case HICCL_MIN: each([](uint32_t x, uint32_t y) { return (uint32_t)min((int)x, (int)y); }); break;
      default: each([](uint32_t x, uint32_t y) { return (x | y) != 0u ? 1u : 0u; }); break;
    }
  }
}

// the sources q .. q + 31 whose tokens are not plain combines, one bit each
__device__ __forceinline__ uint32_t more_than_combine(const uint32_t *tok, uint32_t q, uint32_t nsrc) {
  const uint32_t i = q + (threadIdx.x & 31);
  return __ballot_sync(0xffffffffu, i < nsrc && __ldg(tok + i) != 0u);
}

// One unit of a fold: V vectors of W bytes per lane, at byte offset `off` of
// the lane's first vector, vectors 32 * W bytes apart, those ending past
// `end` left out.  U sources are in flight; every source's token says how it
// enters the accumulator (see TOK_*).  `stack` holds this thread's saved
// values, word k at stack[k * threads].
template <int FAM, int W, int V, int U>
__device__ __forceinline__ void fold_unit(const unsigned long long *__restrict__ P, const uint32_t *__restrict__ tok,
                                          uint32_t nsrc, uint32_t ndst, unsigned long long off, unsigned long long end,
                                          uint32_t dt, uint32_t rop, uint32_t *stack, uint32_t threads) {
  using A = Acc<FAM, W>;
  constexpr int N = A::N;
  uint32_t acc[V * N];
  bool on[V];
#pragma unroll
  for (int v = 0; v < V; ++v) on[v] = off + v * (32 * W) + W <= end;
  static_assert(32 % U == 0, "the sources in flight lie in one 32-bit mask");
  uint32_t sp = 0, nz = 0;   // words saved; which of 32 tokens do more than combine
  for (uint32_t q = 0; q < nsrc; q += U) {
    Raw<W> x[U][V];
    if ((q & 31u) == 0) nz = more_than_combine(tok, q, nsrc);
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (q + u < nsrc) {
        const unsigned long long s = __ldg(P + q + u) + off;
#pragma unroll
        for (int v = 0; v < V; ++v)
          if (on[v]) x[u][v] = ld_raw<W>(s + v * (32 * W));
      }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (q + u < nsrc) {
        auto src = [&](int i) { return A::widen(x[u][i / N], i % N); };
        if (!((nz >> ((q & 31u) + u)) & 1u)) {
          combine<FAM, V * N>(acc, src, dt, rop);
          continue;
        }
        const uint32_t tk = __ldg(tok + q + u);
        if (tk & TOK_START) {
          if (tk & TOK_PUSH) {
#pragma unroll
            for (int i = 0; i < V * N; ++i) stack[(sp + i) * threads] = acc[i];
            sp += V * N;
          }
#pragma unroll
          for (int i = 0; i < V * N; ++i) acc[i] = src(i);
        } else {
          combine<FAM, V * N>(acc, src, dt, rop);
        }
        for (uint32_t o = tk >> TOK_OPS; o; o >>= 2) {
          if ((o & 3u) == TOK_ROUND) {
#pragma unroll
            for (int v = 0; v < V; ++v) A::round(acc + v * N);
            continue;
          }
          sp -= V * N;
          const bool pop = (o & 3u) == TOK_POP;   // the saved value is the left operand
#pragma unroll
          for (int v = 0; v < V; ++v) {
            uint32_t y[N];
#pragma unroll
            for (int i = 0; i < N; ++i) {
              const uint32_t z = stack[(sp + v * N + i) * threads], w = acc[v * N + i];
              acc[v * N + i] = pop ? z : w;
              y[i] = pop ? w : z;
            }
            combine<FAM, N>(acc + v * N, [&](int i) { return y[i]; }, dt, rop);
          }
        }
      }
  }
  Raw<W> r[V];
#pragma unroll
  for (int v = 0; v < V; ++v) r[v] = A::pack(acc + v * N);
#pragma unroll 4
  for (uint32_t d = 0; d < ndst; ++d) {
    const unsigned long long a = __ldg(P + nsrc + d) + off;
#pragma unroll
    for (int v = 0; v < V; ++v)
      if (on[v]) st_raw<W>(a + v * (32 * W), r[v]);
  }
}

template <int W, int V>
__device__ __forceinline__ void copy_unit(const unsigned long long *__restrict__ P, uint32_t ndst,
                                          unsigned long long off, unsigned long long end) {
  Raw<W> r[V];
  bool on[V];
  const unsigned long long s = __ldg(P) + off;
#pragma unroll
  for (int v = 0; v < V; ++v) {
    on[v] = off + v * (32 * W) + W <= end;
    if (on[v]) r[v] = ld_raw<W>(s + v * (32 * W));
  }
#pragma unroll 4
  for (uint32_t d = 0; d < ndst; ++d) {
    const unsigned long long a = __ldg(P + 1 + d) + off;
#pragma unroll
    for (int v = 0; v < V; ++v)
      if (on[v]) st_raw<W>(a + v * (32 * W), r[v]);
  }
}

// the family's fold for a class of any payload but FP8
template <int W, int V, int U>
__device__ __forceinline__ void fold_any(const SweepArgs &A, const SweepClass &k, const unsigned long long *P,
                                         unsigned long long off, unsigned long long end, uint32_t *stack) {
  const uint32_t dt = sweep_dtype(k.meta), rop = sweep_rop(k.meta), threads = blockDim.x;
  const uint32_t *tok = A.toks + k.tok;
  if (dt == HICCL_BF16) {
    if (rop == HICCL_SUM) fold_unit<BF16_SUM, W, V, U>(P, tok, k.nsrc, k.ndst, off, end, dt, rop, stack, threads);
    else fold_unit<BF16_ANY, W, V, U>(P, tok, k.nsrc, k.ndst, off, end, dt, rop, stack, threads);
  } else if constexpr (W >= 4) {
    if (dt == HICCL_F32 && rop == HICCL_SUM)
      fold_unit<F32_SUM, W, V, U>(P, tok, k.nsrc, k.ndst, off, end, dt, rop, stack, threads);
    else fold_unit<ANY_32, W, V, U>(P, tok, k.nsrc, k.ndst, off, end, dt, rop, stack, threads);
  }
}

// ---- units -----------------------------------------------------------------------

// The class and member of a unit; operand pointers at P, the unit's index
// inside the member in `part`.
__device__ __forceinline__ SweepClass find_class(const SweepArgs &A, uint32_t unit, const unsigned long long *&P,
                                                 uint32_t &part) {
  uint32_t lo = 0, hi = A.nclass;
  while (hi - lo > 1) {   // last class whose first unit is not past `unit`
    const uint32_t mid = (lo + hi) >> 1;
    const uint32_t u0 = A.nclass <= SWEEP_PREFIX ? A.unit0[mid] : __ldg(&A.classes[mid].unit0);
    if (u0 <= unit) lo = mid;
    else hi = mid;
  }
  SweepClass k;
  {
    const uint4 *q = reinterpret_cast<const uint4 *>(A.classes + lo);
    uint4 *z = reinterpret_cast<uint4 *>(&k);
#pragma unroll
    for (int i = 0; i < 3; ++i) z[i] = __ldg(q + i);
  }
  const uint32_t at = unit - k.unit0, mem = at / k.upm;
  part = at - mem * k.upm;
  P = A.ptrs + k.ptr + (unsigned long long)mem * (k.nsrc + k.ndst);
  return k;
}

// Launches overlap the previous kernel's tail: the next kernel's CTAs may
// become resident once every CTA of this one has started, and touch nothing
// before this grid has completed.
__device__ __forceinline__ void launch_order() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Where the whole 16-byte vectors of a member lie: all its operands are
// equally far off a boundary, so they start at byte `head` and end at `end`
// of each; the elements before and after are at most 14 + 14 bytes.  (Rows of
// a multiple of 16 bytes with odd chunk lengths are such operands: an odd
// 6 MiB All-reduce over 16 ranks takes 38 us, 55 us by 4-byte accesses.)
struct Body {
  unsigned long long head, end;
};
__device__ __forceinline__ Body body_of(const SweepClass &k, const unsigned long long *P) {
  const unsigned long long h = min((0ull - __ldg(P)) & 15u, k.nbytes);
  return Body{h, h + ((k.nbytes - h) & ~15ull)};
}
// byte offset of this lane's element of W bytes outside the body (nbytes: none)
template <int W>
__device__ __forceinline__ unsigned long long edge_of(const SweepClass &k, const Body &b, int lane) {
  const unsigned long long o = (unsigned long long)lane * W;
  return o < b.head ? o : min(b.end + (o - b.head), k.nbytes);
}

// a copy's unit, and with the last one the member's edges
__device__ __forceinline__ void copy_member(const SweepClass &k, const unsigned long long *P, uint32_t part, int lane) {
  const uint32_t v = sweep_v(k.meta);
  const Body b = body_of(k, P);
  const unsigned long long off = b.head + (unsigned long long)part * 512 * v + lane * 16;
  if (v == 4) copy_unit<16, 4>(P, k.ndst, off, b.end);
  else if (v == 2) copy_unit<16, 2>(P, k.ndst, off, b.end);
  else copy_unit<16, 1>(P, k.ndst, off, b.end);
  if (part + 1 == k.upm && b.end - b.head != k.nbytes) copy_unit<2, 1>(P, k.ndst, edge_of<2>(k, b, lane), k.nbytes);
}

// V vectors a lane in flight, stored to every destination
__global__ void __launch_bounds__(SWEEP_THREADS[SWEEP_COPY], 8) sweep_copy_kernel(const __grid_constant__ SweepArgs A) {
  launch_order();
  const uint32_t unit = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (unit >= A.units) return;
  const unsigned long long *P;
  uint32_t part;
  const SweepClass k = find_class(A, unit, P, part);
  copy_member(k, P, part, threadIdx.x & 31);
}

__global__ void __launch_bounds__(SWEEP_THREADS[SWEEP_FOLD], 8) sweep_fold_kernel(const __grid_constant__ SweepArgs A) {
  extern __shared__ uint32_t saved[];
  launch_order();
  const uint32_t unit = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (unit >= A.units) return;
  const unsigned long long *P;
  uint32_t part;
  const SweepClass k = find_class(A, unit, P, part);
  if (k.nsrc == 1) {
    copy_member(k, P, part, lane);
    return;
  }
  uint32_t *stack = saved + threadIdx.x;
  const uint32_t v = sweep_v(k.meta);
  const Body b = body_of(k, P);
  const unsigned long long off = b.head + (unsigned long long)part * 512 * v + lane * 16;
  if (v == 2) fold_any<16, 2, 8>(A, k, P, off, b.end, stack);
  else fold_any<16, 1, 16>(A, k, P, off, b.end, stack);
  if (part + 1 == k.upm && b.end - b.head != k.nbytes) {
    if (sweep_dtype(k.meta) == HICCL_BF16) fold_any<2, 1, 8>(A, k, P, edge_of<2>(k, b, lane), k.nbytes, stack);
    else fold_any<4, 1, 8>(A, k, P, edge_of<4>(k, b, lane), k.nbytes, stack);
  }
}

// folds of operands that lie differently off a 16-byte boundary: W-byte
// accesses, 4 where every operand and
// the length allow them, else 2
template <int W>
__device__ __forceinline__ void narrow_unit(const SweepArgs &A, const SweepClass &k, const unsigned long long *P,
                                            uint32_t part, int lane, uint32_t *stack) {
  const uint32_t v = sweep_v(k.meta);
  const unsigned long long off = (unsigned long long)part * (32 * W) * v + lane * W;
  if (v == 8) fold_any<W, 8, 4>(A, k, P, off, k.nbytes, stack);
  else if (v == 2) fold_any<W, 2, 8>(A, k, P, off, k.nbytes, stack);
  else fold_any<W, 1, 16>(A, k, P, off, k.nbytes, stack);
}
__global__ void __launch_bounds__(SWEEP_THREADS[SWEEP_NARROW], 10) sweep_narrow_kernel(const __grid_constant__ SweepArgs A) {
  extern __shared__ uint32_t saved[];
  launch_order();
  const uint32_t unit = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (unit >= A.units) return;
  const unsigned long long *P;
  uint32_t part;
  const SweepClass k = find_class(A, unit, P, part);
  if (sweep_lw(k.meta) == 2) narrow_unit<4>(A, k, P, part, lane, saved + threadIdx.x);
  else narrow_unit<2>(A, k, P, part, lane, saved + threadIdx.x);
}

// Copies between operands that lie differently off a 16-byte boundary.  The
// source is read by its aligned vectors; the 16 bytes that a destination's
// vector takes straddle two of them, the lane's own and the next lane's, and
// are shifted out of the pair.  (Element accesses are bound by latency: 64
// bytes a warp request, 90 us for an odd-length BF16 All-to-all of 64 ranks x
// 1 MiB at four requests in flight and 45 us at sixteen, against 27 us here,
// 4.9 TB/s.)  A unit is V rows of 31 destination vectors
// (lane 31 loads only for lane 30) -- 496 source bytes a row; the elements
// that no whole pair covers, at most 31 bytes at each end, go one by one with
// the member's last unit.
__device__ __forceinline__ uint4 shift_pair(const uint4 &a, const uint4 &b, uint32_t e) {
  const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
  const uint32_t bits = 8 * (e & 3u);
  uint4 r;
  auto take = [&](auto c) {
    constexpr int K = decltype(c)::value;
    // (the word past the pair is only reached with bits == 0)
    r.x = __funnelshift_r(w[K], w[K + 1], bits);
    r.y = __funnelshift_r(w[K + 1], w[K + 2], bits);
    r.z = __funnelshift_r(w[K + 2], w[K + 3], bits);
    r.w = __funnelshift_r(w[K + 3], w[K + 4], bits);
  };
  switch (e >> 2) {
    case 0: take(std::integral_constant<int, 0>{}); break;
    case 1: take(std::integral_constant<int, 1>{}); break;
    case 2: take(std::integral_constant<int, 2>{}); break;
    default: take(std::integral_constant<int, 3>{}); break;
  }
  return r;
}
template <int V>
__device__ __forceinline__ void shift_unit(const SweepClass &k, const unsigned long long *P, uint32_t part, int lane) {
  const unsigned long long src = __ldg(P), n = k.nbytes;
  const unsigned long long o0 = (0ull - src) & 15u;           // first whole vector of the source
  const unsigned long long last = o0 + 16 <= n ? o0 + ((n - o0 - 16) & ~15ull) : 0ull;   // the last one
  const unsigned long long base = o0 + ((unsigned long long)part * V * 31 + lane) * 16;
  uint4 a[V], b[V];
  const bool any = o0 + 32 <= n;                              // at least one pair
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const unsigned long long o = base + v * (31 * 16);
    a[v] = make_uint4(0, 0, 0, 0);
    if (any && o <= last) a[v] = __ldcg(reinterpret_cast<const uint4 *>(src + o));
  }
#pragma unroll
  for (int v = 0; v < V; ++v) {
    b[v].x = __shfl_down_sync(0xffffffffu, a[v].x, 1);
    b[v].y = __shfl_down_sync(0xffffffffu, a[v].y, 1);
    b[v].z = __shfl_down_sync(0xffffffffu, a[v].z, 1);
    b[v].w = __shfl_down_sync(0xffffffffu, a[v].w, 1);
  }
  // the ends: lanes 0 .. 15 the first 32 bytes, lanes 16 .. 31 those from the
  // last vector on, two bytes each (a short member has only the first)
  const bool edges = part + 1 == k.upm;
  const unsigned long long at = lane < 16 ? 2ull * lane : (any ? last + 2ull * (lane - 16) : 32 + 2ull * (lane - 16));
  unsigned short ev = 0;
  if (edges && at < n) ev = __ldcg(reinterpret_cast<const unsigned short *>(src + at));
  for (uint32_t d = 0; d < k.ndst; ++d) {
    const unsigned long long dst = __ldg(P + 1 + d);
    const uint32_t e = (uint32_t)((0ull - (dst + o0)) & 15u);   // from a source vector to the destination's
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const unsigned long long o = base + v * (31 * 16);
      if (any && lane < 31 && o < last) *reinterpret_cast<uint4 *>(dst + o + e) = shift_pair(a[v], b[v], e);
    }
    if (edges && at < n && (!any || (lane < 16 ? at < o0 + e : at >= last + e)))
      *reinterpret_cast<unsigned short *>(dst + at) = ev;
  }
}
__global__ void __launch_bounds__(SWEEP_THREADS[SWEEP_SHIFT], 8) sweep_shift_kernel(const __grid_constant__ SweepArgs A) {
  launch_order();
  const uint32_t unit = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (unit >= A.units) return;
  const unsigned long long *P;
  uint32_t part;
  const SweepClass k = find_class(A, unit, P, part);
  if (sweep_v(k.meta) == 4) shift_unit<4>(k, P, part, threadIdx.x & 31);
  else shift_unit<1>(k, P, part, threadIdx.x & 31);
}

// ---- FP8 blocks --------------------------------------------------------------------
// A group of 8 lanes folds one 144-byte block, lane `sub` owning codes
// 16 * sub .. 16 * sub + 15; four blocks a warp.

struct Fp8Raw {
  uint4 c;
  float scale;
};

// two binary32 values in one 64-bit register pair
__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
  unsigned long long d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ void unpack2(unsigned long long d, float &lo, float &hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(d));
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// rounded products: fma with -0, which a kernel argument supplies so that the
// product is not contracted into the add that follows it
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b,
                                                   unsigned long long minus0) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(minus0));
  return d;
}

// the 16 values of a lane, code x scale
__device__ __forceinline__ void fp8_widen(const Fp8Raw &x, unsigned long long minus0, unsigned long long *v) {
  const uint32_t w[4] = {x.c.x, x.c.y, x.c.z, x.c.w};
  const unsigned long long s = pack2(x.scale, x.scale);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float4 f = e4m3x4_to_f32x4(w[j]);
    v[2 * j] = mul2(pack2(f.x, f.y), s, minus0);
    v[2 * j + 1] = mul2(pack2(f.z, f.w), s, minus0);
  }
}
// a fresh scale amax / 448 and codes of value x (448 / amax) (both factors 1
// when amax is 0); all lanes of the warp take part
__device__ __forceinline__ Fp8Raw fp8_encode(const unsigned long long *v) {
  float acc[16];
#pragma unroll
  for (int i = 0; i < 8; ++i) unpack2(v[i], acc[2 * i], acc[2 * i + 1]);
  float amax = 0.f;
#pragma unroll
  for (int i = 0; i < 16; ++i) amax = fmaxf(amax, fabsf(acc[i]));
  amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 1));
  amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 2));
  amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 4));
  Fp8Raw r;
  r.scale = amax > 0.f ? __fdiv_rn(amax, 448.f) : 1.f;
  const float inv = amax > 0.f ? __fdiv_rn(448.f, amax) : 1.f;
  uint32_t w[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t lo = f32x2_to_e4m3x2(__fmul_rn(acc[4 * i], inv), __fmul_rn(acc[4 * i + 1], inv));
    const uint32_t hi = f32x2_to_e4m3x2(__fmul_rn(acc[4 * i + 2], inv), __fmul_rn(acc[4 * i + 3], inv));
    w[i] = lo | (hi << 16);
  }
  r.c = make_uint4(w[0], w[1], w[2], w[3]);
  return r;
}

constexpr int FP8_SLOTS = 8;                                    // sources a warp keeps in flight
constexpr uint32_t FP8_STEP = 4 * FP8_BLOCK_BYTES;              // bytes of a source in one slot

__device__ __forceinline__ void cp_async16(uint32_t dst, unsigned long long src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// A unit is four blocks, 576 bytes of every operand.  A source takes about 100
// instructions, so a warp is busy while its loads should fly; they
// pass through a ring of slots in shared memory, one asynchronous copy group
// a source, which keeps FP8_SLOTS - 1 in flight through folds, encodings and
// stores without holding registers (72 a thread, 24 warps an SM).  Copies and
// stores move the unit as one range of whole sectors, and only the fold reads
// it by blocks.  All-reduce of 16 Mi values a rank over 32 ranks ({4, 8}),
// 1.21 GB in and out: 265 us with the next sources loaded into registers (16
// warps an SM; 403 us when refilled one by one), 223 us through the ring by
// blocks, 199 us by the unit's range, 6.1 TB/s; two or four units a warp
// lose 5 and 10 %, neighbouring warps on neighbouring units read longer
// stretches of each source at a time.
__global__ void __launch_bounds__(SWEEP_THREADS[SWEEP_FP8], 6) sweep_fp8_kernel(const __grid_constant__ SweepArgs A) {
  extern __shared__ __align__(16) uint32_t saved[];
  launch_order();
  const uint32_t unit = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (unit >= A.units) return;
  const unsigned long long *P;
  uint32_t part;
  const SweepClass k = find_class(A, unit, P, part);
  const uint32_t *tok = A.toks + k.tok;
  const uint32_t threads = blockDim.x, sub = lane & 7;
  const unsigned long long minus0 = A.minus0;
  char *ring = reinterpret_cast<char *>(saved) + (threadIdx.x >> 5) * (FP8_SLOTS * FP8_STEP);
  char *mine = ring + (lane >> 3) * FP8_BLOCK_BYTES;   // this group's block in slot 0
  const uint32_t ring_at = static_cast<uint32_t>(__cvta_generic_to_shared(ring)) + 16 * lane;
  float *stack = reinterpret_cast<float *>(saved) + (threads >> 5) * (FP8_SLOTS * FP8_STEP / 4) + threadIdx.x;

  // this lane's 16 bytes of the unit, and (lanes 0 .. 3) 16 of its last 64
  const unsigned long long off = (unsigned long long)part * FP8_STEP + 16 * lane;
  const bool on = off < k.nbytes, on2 = lane < 4 && off + 512 < k.nbytes;
  unsigned long long lptr = __ldg(P);   // of source lq
  uint32_t lq = 0;
  auto load = [&](int slot) {
    if (lq < k.nsrc) {
      const unsigned long long s = lptr + off;
      if (on) cp_async16(ring_at + slot * FP8_STEP, s);
      if (on2) cp_async16(ring_at + slot * FP8_STEP + 512, s + 512);
      if (++lq < k.nsrc) lptr = __ldg(P + lq);
    }
    cp_commit();
  };
#pragma unroll
  for (int u = 0; u < FP8_SLOTS - 1; ++u) load(u);
  unsigned long long acc[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] = 0ull;
  uint32_t sp = 0, nz = 0;   // words saved; which of 32 tokens do more than combine
  uint32_t slot = 0;
  for (uint32_t q = 0; q < k.nsrc; ++q) {
    if ((q & 31u) == 0) nz = more_than_combine(tok, q, k.nsrc);
    cp_wait<FP8_SLOTS - 2>();
    __syncwarp();              // every lane's copies have landed, and the slot read last is free
    load((slot + FP8_SLOTS - 1) % FP8_SLOTS);
    Fp8Raw x;
    x.c = *reinterpret_cast<const uint4 *>(mine + slot * FP8_STEP + 16 * sub);
    x.scale = *reinterpret_cast<const float *>(mine + slot * FP8_STEP + 128);
    slot = (slot + 1) % FP8_SLOTS;
    unsigned long long y[8];
    fp8_widen(x, minus0, y);
    if (!((nz >> (q & 31u)) & 1u)) {
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i] = add2(acc[i], y[i]);
      continue;
    }
    const uint32_t tk = __ldg(tok + q);
    if (tk & TOK_START) {
      if (tk & TOK_PUSH) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          float lo, hi;
          unpack2(acc[i], lo, hi);
          stack[(sp + 2 * i) * threads] = lo;
          stack[(sp + 2 * i + 1) * threads] = hi;
        }
        sp += 16;
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i] = y[i];
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i] = add2(acc[i], y[i]);
    }
    for (uint32_t o = tk >> TOK_OPS; o; o >>= 2) {
      if ((o & 3u) == TOK_ROUND) {
        fp8_widen(fp8_encode(acc), minus0, acc);
      } else {
        sp -= 16;
#pragma unroll
        for (int i = 0; i < 8; ++i) {   // (a sum of two is the same in both orders)
          const float lo = stack[(sp + 2 * i) * threads], hi = stack[(sp + 2 * i + 1) * threads];
          acc[i] = add2(pack2(lo, hi), acc[i]);
        }
      }
    }
  }
  const Fp8Raw r = fp8_encode(acc);
  cp_wait<0>();
  __syncwarp();   // the ring is free: the result takes slot 0
  *reinterpret_cast<uint4 *>(mine + 16 * sub) = r.c;
  if (sub == 0) *reinterpret_cast<uint4 *>(mine + 128) = make_uint4(__float_as_uint(r.scale), 0u, 0u, 0u);
  __syncwarp();
  const uint4 v = *reinterpret_cast<const uint4 *>(ring + 16 * lane);
  const uint4 v2 = *reinterpret_cast<const uint4 *>(ring + 512 + 16 * (lane & 3));
#pragma unroll 4
  for (uint32_t d = 0; d < k.ndst; ++d) {
    const unsigned long long a = __ldg(P + k.nsrc + d) + off;
    if (on) *reinterpret_cast<uint4 *>(a) = v;
    if (on2) *reinterpret_cast<uint4 *>(a + 512) = v2;
  }
}

typedef void (*Kernel)(const SweepArgs);
const Kernel KERNELS[SWEEP_KERNELS] = {sweep_copy_kernel, sweep_fold_kernel, sweep_fp8_kernel, sweep_narrow_kernel,
                                         sweep_shift_kernel};

}  // namespace

// dynamic shared memory: at most SWEEP_MAX_DEPTH values of 16 words for each
// of 128 threads and four rings, or of 16 words for 256; more than half an SM's keeps a second CTA
// off it
constexpr size_t SWEEP_MAX_SMEM = SWEEP_MAX_DEPTH * 16 * 4 * 256 + 8 * FP8_SLOTS * FP8_STEP, SWEEP_HALF_SM = 120 * 1024;

cudaError_t sweep_prepare() {
  for (uint32_t i = 0; i < SWEEP_KERNELS; ++i) {
    const cudaError_t e = cudaFuncSetAttribute(KERNELS[i], cudaFuncAttributeMaxDynamicSharedMemorySize, SWEEP_MAX_SMEM);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t sweep_launch(const SweepLaunch &L, const SweepArgs &A, bool one_per_sm, cudaStream_t s) {
  const unsigned warps = L.threads / 32;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((L.units + warps - 1) / warps);
  cfg.blockDim = dim3(L.threads);
  cfg.dynamicSmemBytes = (size_t)L.stack_words * 4 * L.threads;
  if (L.kernel == SWEEP_FP8) cfg.dynamicSmemBytes += warps * FP8_SLOTS * FP8_STEP;
  if (one_per_sm && cfg.dynamicSmemBytes < SWEEP_HALF_SM) cfg.dynamicSmemBytes = SWEEP_HALF_SM;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, KERNELS[L.kernel], A);
}

}  // namespace hiccl
