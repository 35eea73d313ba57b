// Sweep kernels: a program's expressions evaluated in one pass over its
// outputs (hiccl_sweep.cpp builds the classes; see there for why this equals
// the factorized schedule).
//
// What bounds a pass is memory: every input is read once and every output
// written once, with at most one add per value between.  A warp takes one
// unit of one member.  Folds bring their sources through a ring of
// asynchronous copies in shared memory, one 16-byte vector a lane and source,
// so that the loads in flight (30 warps x 4 to 6 KiB an SM) need no registers
// and never wait for a fold; copies load up to four vectors a lane.  The
// value goes to its destinations straight from registers.  Nothing waits on
// another CTA, so the grid is one warp per unit, in CTAs of two to four warps
// that free their SM as they finish, and the hardware's CTA scheduler
// balances the tail.  Measured against: a persistent grid of the same code,
// 74 against 41 us for a 4 MiB Broadcast to 64 ranks; bulk (TMA) loads and
// stores through shared-memory rings, 672 against 624 us for the All-reduce
// below; eight sources in registers, 53.9 against 46.7 us for a BF16
// Reduce-scatter of 16 ranks x 16 MiB.
//
// Against the step executor, GB300, a start as a program times it: All-reduce
// of 64 MiB a rank over 32 ranks 768 -> 635 us (623 us, 6.89 TB/s of the
// inputs read and outputs written once, without the host), All-reduce of 64
// KiB of BF16 over 8 ranks (graph replay) 22.9 -> 6.2 us, the seven
// collectives of 64 ranks x 4 MiB (graph replay) 455 -> 290 us, an odd-length
// 6 MiB All-reduce over 16 ranks 525 -> 45 us.

#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "hiccl_device.cuh"
#include "hiccl_internal.h"
#include "hiccl_sweep.h"

namespace hiccl {

namespace {

// Groups of a fold's ring: three hold 6 KiB a warp, 30 warps an SM.  A pass
// with fewer units than half of those warps (SHORT_UNITS) deepens it instead
// (a 64-way int32 maximum of 1 MiB a rank, 2048 units: 15.1 us with three,
// 13.7 us with five).  Measured with two / three / four groups: 45.1 / 43.6 /
// 50 us for a Reduce-scatter of 64 ranks x 4 MiB, 48.7 / 46.7 / 56 us for 16
// ranks x 16 MiB of BF16.
constexpr int FOLD_GROUPS = 3, FOLD_GROUPS_SHORT = 5;
constexpr uint32_t SHORT_UNITS = SWEEP_SMS * 16;

// ---- units -----------------------------------------------------------------------

// What a unit does: part `part` of a member of class k with operand pointers
// P, stored to the destinations P[d0 .. d1).
struct Unit {
  SweepClass k;
  const unsigned long long *P;
  uint32_t part, d0, d1;
};
__device__ __forceinline__ Unit find_unit(const SweepArgs &A, uint32_t unit) {
  uint32_t lo = 0, hi = A.nclass;
  if (hi > SWEEP_PREFIX) {
    lo = __ldg(A.hints + (unit >> SWEEP_HINT_SHIFT));
    hi = __ldg(A.hints + (unit >> SWEEP_HINT_SHIFT) + 1) + 1;
  }
  while (hi - lo > 1) {   // last class whose first unit is not past `unit`
    const uint32_t mid = (lo + hi) >> 1;
    const uint32_t u0 = A.nclass <= SWEEP_PREFIX ? A.unit0[mid] : __ldg(&A.classes[mid].unit0);
    if (u0 <= unit) lo = mid;
    else hi = mid;
  }
  Unit r;
  if (A.nclass <= SWEEP_INLINE) {
    r.k = A.first[lo];
  } else {
    const uint4 *q = reinterpret_cast<const uint4 *>(A.classes + lo);
    uint4 *z = reinterpret_cast<uint4 *>(&r.k);
#pragma unroll
    for (int i = 0; i < 4; ++i) z[i] = __ldg(q + i);
  }
  const SweepClass &k = r.k;
  uint32_t at = unit - k.unit0, g = 0;
  if (k.group < k.ndst) {   // destination groups, tile by tile of the source
    const uint32_t all = k.upm * k.nmem, tile = SWEEP_TILE / sweep_v(k.meta);
    uint32_t base = 0, cur = all;
    if (all > tile) {
      const unsigned long long per = (unsigned long long)tile * ((k.ndst + k.group - 1) / k.group);
      const uint32_t t = (uint32_t)(at / per);
      at -= (uint32_t)(t * per);
      base = t * tile;
      cur = min(tile, all - base);
    }
    g = at / cur;
    at = base + (at - g * cur);
  }
  const uint32_t mem = at / k.upm;
  r.part = at - mem * k.upm;
  r.P = A.ptrs + k.ptr + (unsigned long long)mem * (k.nsrc + k.ndst);
  r.d0 = k.nsrc + g * k.group;
  r.d1 = k.nsrc + min(k.ndst, (g + 1) * k.group);
  return r;
}

// ---- accesses of W bytes per lane ----------------------------------------------

template <int W>
struct Raw {
  uint32_t w[W >= 4 ? W / 4 : 1];
};
// (L2 only: under programmatic launch another kernel may just have written
// these lines, and no SM reads a line twice)
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

// a[i] = a[i] op b(i) over N words of S sources in turn (source j's are
// b(j * N) ..), the operator's branch taken once for all of them
template <int FAM, int N, int S = 1, typename F>
__device__ __forceinline__ void combine(uint32_t *a, F b, uint32_t dt, uint32_t rop) {
  auto f = [](uint32_t x) { return __uint_as_float(x); };
  auto each = [&](auto op) {
#pragma unroll
    for (int i = 0; i < N * S; ++i) a[i % N] = op(a[i % N], b(i));
  };
  auto add = [&](uint32_t x, uint32_t y) { return __float_as_uint(__fadd_rn(f(x), f(y))); };
  auto fmx = [&](uint32_t x, uint32_t y) { return __float_as_uint(fmaxf(f(x), f(y))); };
  auto fmn = [&](uint32_t x, uint32_t y) { return __float_as_uint(fminf(f(x), f(y))); };
  if constexpr ((FAM == F32_SUM || FAM == BF16_SUM) && N % 2 == 0) {
#pragma unroll
    for (int j = 0; j < N * S; j += 2) {   // two sums an instruction
      const int i = j % N;
      float lo, hi;
      unpack2(add2(pack2(f(a[i]), f(a[i + 1])), pack2(f(b(j)), f(b(j + 1)))), lo, hi);
      a[i] = __float_as_uint(lo);
      a[i + 1] = __float_as_uint(hi);
    }
  } else if constexpr (FAM == F32_SUM || FAM == BF16_SUM) {
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

// The tokens of 32 sources, one a lane: a bit for each that is not a plain
// combine, and the token itself on request.
struct Tokens {
  uint32_t mine = 0, nz = 0;
  __device__ __forceinline__ void read(const uint32_t *tok, uint32_t q, uint32_t nsrc) {   // q a multiple of 32
    const uint32_t i = q + (threadIdx.x & 31);
    mine = i < nsrc ? __ldg(tok + i) : 0u;
    nz = __ballot_sync(0xffffffffu, mine != 0u);
  }
  __device__ __forceinline__ bool plain(uint32_t q) const { return !((nz >> (q & 31u)) & 1u); }
  __device__ __forceinline__ bool plain4(uint32_t q) const { return !((nz >> (q & 31u)) & 15u); }
  __device__ __forceinline__ uint32_t at(uint32_t q) const { return __shfl_sync(0xffffffffu, mine, q & 31u); }
};

// The value of an expression of nsrc sources: V vectors of W bytes a lane,
// load(q, x) filling source q's.  U sources are in flight; every source's
// token says how it enters the accumulator (see TOK_*).  `stack` holds this
// thread's saved values, word k at stack[k * threads].
template <int FAM, int W, int V, int U, typename LD>
__device__ __forceinline__ void fold_value(LD load, const uint32_t *__restrict__ tok, uint32_t nsrc, uint32_t dt,
                                           uint32_t rop, uint32_t *stack, uint32_t threads, Raw<W> (&r)[V]) {
  using A = Acc<FAM, W>;
  constexpr int N = A::N;
  uint32_t acc[V * N];
  static_assert(32 % U == 0, "the sources in flight lie in one 32-bit mask");
  uint32_t sp = 0;   // words saved
  Tokens t;
  for (uint32_t q = 0; q < nsrc; q += U) {
    Raw<W> x[U][V];
    if ((q & 31u) == 0) t.read(tok, q, nsrc);
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (q + u < nsrc) load(q + u, x[u]);
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (q + u < nsrc) {
        auto src = [&](int i) { return A::widen(x[u][i / N], i % N); };
        if (t.plain(q + u)) {
          combine<FAM, V * N>(acc, src, dt, rop);
          continue;
        }
        const uint32_t tk = t.at(q + u);
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
#pragma unroll
          for (int v = 0; v < V; ++v)
            combine<FAM, N>(acc + v * N, [&](int i) { return stack[(sp + v * N + i) * threads]; }, dt, rop);
        }
      }
  }
#pragma unroll
  for (int v = 0; v < V; ++v) r[v] = A::pack(acc + v * N);
}

// One unit of a fold: the lane's first vector at byte offset `off` of every
// operand, vectors 32 * W bytes apart, those ending past `end` left out.
template <int FAM, int W, int V, int U>
__device__ __forceinline__ void fold_unit(const unsigned long long *__restrict__ P, const uint32_t *__restrict__ tok,
                                          uint32_t nsrc, uint32_t ndst, unsigned long long off, unsigned long long end,
                                          uint32_t dt, uint32_t rop, uint32_t *stack, uint32_t threads) {
  bool on[V];
#pragma unroll
  for (int v = 0; v < V; ++v) on[v] = off + v * (32 * W) + W <= end;
  Raw<W> r[V];
  fold_value<FAM, W, V, U>(
      [&](uint32_t q, Raw<W> (&x)[V]) {
        const unsigned long long s = __ldg(P + q) + off;
#pragma unroll
        for (int v = 0; v < V; ++v)
          if (on[v]) x[v] = ld_raw<W>(s + v * (32 * W));
      },
      tok, nsrc, dt, rop, stack, threads, r);
#pragma unroll 4
  for (uint32_t d = 0; d < ndst; ++d) {
    const unsigned long long a = __ldg(P + nsrc + d) + off;
#pragma unroll
    for (int v = 0; v < V; ++v)
      if (on[v]) st_raw<W>(a + v * (32 * W), r[v]);
  }
}

// V vectors of the source at P[0] to the destinations P[d0 .. d1)
template <int W, int V>
__device__ __forceinline__ void copy_unit(const unsigned long long *__restrict__ P, uint32_t d0, uint32_t d1,
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
  for (uint32_t d = d0; d < d1; ++d) {
    const unsigned long long a = __ldg(P + d) + off;
#pragma unroll
    for (int v = 0; v < V; ++v)
      if (on[v]) st_raw<W>(a + v * (32 * W), r[v]);
  }
}

__device__ __forceinline__ void cp_async16(uint32_t dst, unsigned long long src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// pointer q of a list of n that the warp reads 32 at a time, lane i holding
// the i-th of the block that q lies in; every lane takes part.  (The rings
// leave so little L1 that a load per pointer goes to L2: 57 instead of 51 us
// for a BF16 Reduce-scatter of 16 ranks x 16 MiB.)
__device__ __forceinline__ unsigned long long pointer_at(const unsigned long long *P, uint32_t q, uint32_t n,
                                                         unsigned long long &held) {
  const uint32_t lane = threadIdx.x & 31;
  if ((q & 31u) == 0) held = q + lane < n ? __ldg(P + q + lane) : 0ull;
  return __shfl_sync(0xffffffffu, held, q & 31u);
}

// One unit of a fold of 16-byte vectors, one per lane at byte offset `off`.
// Sources pass through a ring of G groups of RING_GROUP slots of the warp, an
// asynchronous copy group each, so that G - 1 groups stay in flight without
// registers for them.  (Waiting and committing takes about 250 cycles; per
// source, not per group, it was most of the 366 a source took.)
constexpr uint32_t RING_GROUP = 4;
static_assert(32 % RING_GROUP == 0, "a group lies in one block of 32 sources");

template <int FAM, int G>
__device__ __forceinline__ void fold_ring(const SweepArgs &A, const Unit &u, unsigned long long off, bool on,
                                          uint32_t dt, uint32_t rop, char *ring, uint4 *stack, uint32_t threads) {
  using C = Acc<FAM, 16>;
  constexpr int N = C::N;
  const SweepClass &k = u.k;
  const uint32_t *tok = A.toks + k.tok;
  const uint32_t ring_at = static_cast<uint32_t>(__cvta_generic_to_shared(ring));
  unsigned long long held = 0;
  uint32_t lq = 0;   // next source to load
  auto load = [&](uint32_t g) {
#pragma unroll
    for (uint32_t i = 0; i < RING_GROUP; ++i)
      if (lq + i < k.nsrc) {
        const unsigned long long s = pointer_at(u.P, lq + i, k.nsrc, held) + off;
        if (on) cp_async16(ring_at + (g * RING_GROUP + i) * 512, s);
      }
    lq += RING_GROUP;
    cp_commit();
  };
#pragma unroll 1
  for (uint32_t g = 0; g < G - 1; ++g) load(g);
  uint32_t acc[N];
  uint32_t sp = 0;   // saved values end here
  Tokens t;
  uint32_t g = 0;
#pragma unroll 1
  for (uint32_t q = 0; q < k.nsrc; q += RING_GROUP) {
    if ((q & 31u) == 0) t.read(tok, q, k.nsrc);
    cp_wait<G - 2>();
    load(g == 0 ? G - 1 : g - 1);   // the group read last
    Raw<16> x[RING_GROUP];
#pragma unroll
    for (uint32_t i = 0; i < RING_GROUP; ++i) {
      const uint4 v = *reinterpret_cast<const uint4 *>(ring + (g * RING_GROUP + i) * 512);
      x[i].w[0] = v.x;
      x[i].w[1] = v.y;
      x[i].w[2] = v.z;
      x[i].w[3] = v.w;
    }
    if (++g == G) g = 0;
    // A group of plain combines takes its operator's branch once: the chain of
    // tests between sources bounds a short pass (a 64-way int32 maximum of 1 MiB
    // a rank 17.4 -> 13.7 us).  Sums have no such branch and would only pay for
    // a second copy of the loop in registers (spills, 2 to 4 % slower).
    static_assert(RING_GROUP == 4, "plain4");
    if constexpr (FAM == ANY_32 || FAM == BF16_ANY)
      if (q + RING_GROUP <= k.nsrc && t.plain4(q)) {
        combine<FAM, N, RING_GROUP>(acc, [&](int j) { return C::widen(x[j / N], j % N); }, dt, rop);
        continue;
      }
#pragma unroll
    for (uint32_t i = 0; i < RING_GROUP; ++i) {
      auto src = [&](int j) { return C::widen(x[i], j); };
      if (q + i >= k.nsrc) break;
      if (t.plain(q + i)) {
        combine<FAM, N>(acc, src, dt, rop);
        continue;
      }
      const uint32_t tk = t.at(q + i);
      if (tk & TOK_START) {
        if (tk & TOK_PUSH) {
#pragma unroll
          for (int j = 0; j < N; j += 4, sp += threads)
            stack[sp] = make_uint4(acc[j], acc[j + 1], acc[j + 2], acc[j + 3]);
        }
#pragma unroll
        for (int j = 0; j < N; ++j) acc[j] = src(j);
      } else {
        combine<FAM, N>(acc, src, dt, rop);
      }
      for (uint32_t o = tk >> TOK_OPS; o; o >>= 2) {
        if ((o & 3u) == TOK_ROUND) {
          C::round(acc);
          continue;
        }
        sp -= threads * (N / 4);
        uint32_t y[N];
#pragma unroll
        for (int j = 0; j < N; j += 4) {
          const uint4 z = stack[sp + j / 4 * threads];
          y[j] = z.x;
          y[j + 1] = z.y;
          y[j + 2] = z.z;
          y[j + 3] = z.w;
        }
        combine<FAM, N>(acc, [&](int j) { return y[j]; }, dt, rop);
      }
    }
  }
  const Raw<16> r = C::pack(acc);
#pragma unroll 4
  for (uint32_t d = 0; d < k.ndst; ++d) {
    const unsigned long long a = pointer_at(u.P + k.nsrc, d, k.ndst, held) + off;
    if (on) st_raw<16>(a, r);
  }
}

// the family's fold for a class of any payload but FP8
template <int W, int V, int U>
__device__ __forceinline__ void fold_any(const SweepArgs &A, const SweepClass &k, const unsigned long long *P,
                                         unsigned long long off, unsigned long long end, uint32_t *stack,
                                         uint32_t threads) {
  const uint32_t dt = sweep_dtype(k.meta), rop = sweep_rop(k.meta);
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

// Launches overlap the previous kernel's tail: the next kernel's CTAs may
// become resident once every CTA of this one has started, and touch nothing
// before this grid has completed.
__device__ __forceinline__ void launch_order() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Where the whole 16-byte vectors of a member lie: all its operands are
// equally far off a boundary (of 32 bytes where they agree that far, so that no
// sector is written by two warps), so they start at byte `head` and end at
// `end` of each; the elements before and after are at most 30 + 14 bytes.  (Rows of
// a multiple of 16 bytes with odd chunk lengths are such operands: an odd
// 6 MiB All-reduce over 16 ranks takes 36 us, 38 us from 16-byte boundaries
// and 55 us by 4-byte accesses.)
struct Body {
  unsigned long long head, end;
};
__device__ __forceinline__ Body body_of(const SweepClass &k, const unsigned long long *P) {
  const unsigned long long h = min((0ull - __ldg(P)) & ((1u << sweep_lw(k.meta)) - 1u), k.nbytes);
  return Body{h, h + ((k.nbytes - h) & ~15ull)};
}
// byte offset of this lane's element of W bytes outside the body (nbytes: none)
template <int W>
__device__ __forceinline__ unsigned long long edge_of(const SweepClass &k, const Body &b, int lane) {
  const unsigned long long o = (unsigned long long)lane * W;
  return o < b.head ? o : min(b.end + (o - b.head), k.nbytes);
}

// a copy's unit, and with the last one the member's edges
__device__ __forceinline__ void copy_member(const Unit &u, int lane) {
  const SweepClass &k = u.k;
  const uint32_t v = sweep_v(k.meta);
  const Body b = body_of(k, u.P);
  const unsigned long long off = b.head + (unsigned long long)u.part * 512 * v + lane * 16;
  if (v == 4) copy_unit<16, 4>(u.P, u.d0, u.d1, off, b.end);
  else if (v == 2) copy_unit<16, 2>(u.P, u.d0, u.d1, off, b.end);
  else copy_unit<16, 1>(u.P, u.d0, u.d1, off, b.end);
  if (u.part + 1 == k.upm && b.end - b.head != k.nbytes)
    copy_unit<2, 1>(u.P, u.d0, u.d1, edge_of<2>(k, b, lane), k.nbytes);
}

// The units of a warp: one, in a grid that has a warp for each; or (WALK) every
// so many, in a grid of one CTA an SM.
template <bool WALK, typename F>
__device__ __forceinline__ void each_unit(const SweepArgs &A, F body) {
  const uint32_t unit = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if constexpr (WALK) {
    const uint32_t step = gridDim.x * (blockDim.x >> 5);
#pragma unroll 1
    for (unsigned long long i = unit; i < A.units; i += step) body((uint32_t)i);
  } else {
    if (unit < A.units) body(unit);
  }
}
// ONE: the kernel for one CTA an SM
#define SWEEP_BOUNDS(kern, ctas) __launch_bounds__(ONE ? SWEEP_ONE_THREADS : SWEEP_THREADS[kern], ONE ? 1 : ctas)

// V vectors a lane in flight, stored to a group of destinations
template <bool ONE>
__global__ void SWEEP_BOUNDS(SWEEP_COPY, 8) sweep_copy_kernel(const __grid_constant__ SweepArgs A) {
  launch_order();
  each_unit<ONE>(A, [&](uint32_t unit) { copy_member(find_unit(A, unit), threadIdx.x & 31); });
}

template <int G>
__device__ __forceinline__ void fold_member(const SweepArgs &A, const Unit &u, int lane) {
  extern __shared__ __align__(16) uint32_t saved[];
  const SweepClass &k = u.k;
  const uint32_t dt = sweep_dtype(k.meta), rop = sweep_rop(k.meta), threads = blockDim.x;
  char *ring = reinterpret_cast<char *>(saved) + (threadIdx.x >> 5) * (G * RING_GROUP * 512) + lane * 16;
  uint4 *stack = reinterpret_cast<uint4 *>(saved) + (threads >> 5) * (G * RING_GROUP * 32) + threadIdx.x;   // saved values
  const Body b = body_of(k, u.P);
  const unsigned long long off = b.head + (unsigned long long)u.part * 512 + lane * 16;
  const bool on = off + 16 <= b.end;
  if (dt == HICCL_BF16) {
    if (rop == HICCL_SUM) fold_ring<BF16_SUM, G>(A, u, off, on, dt, rop, ring, stack, threads);
    else fold_ring<BF16_ANY, G>(A, u, off, on, dt, rop, ring, stack, threads);
  } else {
    if (dt == HICCL_F32 && rop == HICCL_SUM) fold_ring<F32_SUM, G>(A, u, off, on, dt, rop, ring, stack, threads);
    else fold_ring<ANY_32, G>(A, u, off, on, dt, rop, ring, stack, threads);
  }
  if (u.part + 1 == k.upm && b.end - b.head != k.nbytes) {
    uint32_t *words = reinterpret_cast<uint32_t *>(stack);   // one of each of this thread's own vectors
    if (dt == HICCL_BF16) fold_any<2, 1, 8>(A, k, u.P, edge_of<2>(k, b, lane), k.nbytes, words, 4 * threads);
    else fold_any<4, 1, 8>(A, k, u.P, edge_of<4>(k, b, lane), k.nbytes, words, 4 * threads);
  }
}
template <bool ONE>
__global__ void SWEEP_BOUNDS(SWEEP_FOLD, 16) sweep_fold_kernel(const __grid_constant__ SweepArgs A) {
  launch_order();
  each_unit<false>(A, [&](uint32_t unit) {
    const int lane = threadIdx.x & 31;
    const Unit u = find_unit(A, unit);
    if (u.k.nsrc == 1) copy_member(u, lane);
    else if (A.groups == FOLD_GROUPS) fold_member<FOLD_GROUPS>(A, u, lane);
    else fold_member<FOLD_GROUPS_SHORT>(A, u, lane);
  });
}

// A short fold pass: a CTA to a unit.  Its warps evaluate the expression's
// sections (SweepClass::team), leave their values in shared memory, and after
// a barrier every warp evaluates the expression of those and stores its share
// of the destinations.
template <int FAM, int W>
__device__ __forceinline__ void team_unit(const SweepArgs &A, const Unit &u, unsigned long long off,
                                          unsigned long long end, uint32_t dt, uint32_t rop, uint4 *parts,
                                          uint32_t *stack) {
  const SweepClass &k = u.k;
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const uint32_t *tok = A.toks + k.ttok, *bounds = tok + k.nsrc, *upper = bounds + k.team + 1;
  const bool on = off + W <= end;
  auto part = [&](uint32_t s) { return reinterpret_cast<Raw<W> *>(parts + s * 32 + lane); };
  Raw<W> r[1];
  for (uint32_t s = warp; s < k.team; s += warps) {
    const uint32_t q0 = __ldg(bounds + s), q1 = __ldg(bounds + s + 1);
    fold_value<FAM, W, 1, 8>(
        [&](uint32_t q, Raw<W> (&x)[1]) {
          const unsigned long long a = __ldg(u.P + q0 + q) + off;
          if (on) x[0] = ld_raw<W>(a);
        },
        tok + q0, q1 - q0, dt, rop, stack, blockDim.x, r);
    *part(s) = r[0];
  }
  __syncthreads();
  fold_value<FAM, W, 1, 8>([&](uint32_t s, Raw<W> (&x)[1]) { x[0] = *part(s); }, upper, k.team, dt, rop, stack,
                           blockDim.x, r);
  if (!on) return;
#pragma unroll 4
  for (uint32_t d = warp; d < k.ndst; d += warps) st_raw<W>(__ldg(u.P + k.nsrc + d) + off, r[0]);
}
template <int W>
__device__ __forceinline__ void team_any(const SweepArgs &A, const Unit &u, unsigned long long off,
                                         unsigned long long end, uint4 *parts, uint32_t *stack) {
  const uint32_t dt = sweep_dtype(u.k.meta), rop = sweep_rop(u.k.meta);
  if (dt == HICCL_BF16) {
    if (rop == HICCL_SUM) team_unit<BF16_SUM, W>(A, u, off, end, dt, rop, parts, stack);
    else team_unit<BF16_ANY, W>(A, u, off, end, dt, rop, parts, stack);
  } else if constexpr (W >= 4) {
    if (dt == HICCL_F32 && rop == HICCL_SUM) team_unit<F32_SUM, W>(A, u, off, end, dt, rop, parts, stack);
    else team_unit<ANY_32, W>(A, u, off, end, dt, rop, parts, stack);
  }
}
// (MANY: more than SWEEP_TEAM_STATIC sections, whose values then lie in dynamic shared
// memory; with all of them there, small passes take 0.2 to 0.4 us longer, 4.5
// instead of 4.1 us for a maximum over 8 ranks)
template <bool MANY>
__global__ void __launch_bounds__(SWEEP_THREADS[SWEEP_TEAM], 2)
    sweep_team_kernel(const __grid_constant__ SweepArgs A) {
  __shared__ uint4 few[MANY ? 1 : SWEEP_TEAM_STATIC * 32];
  extern __shared__ __align__(16) uint32_t saved[];
  launch_order();
  const int lane = threadIdx.x & 31;
  const Unit u = find_unit(A, blockIdx.x);
  uint4 *parts = MANY ? reinterpret_cast<uint4 *>(saved) : few;
  uint32_t *stack = saved + (MANY ? A.sections * 128 : 0) + threadIdx.x;
  const Body b = body_of(u.k, u.P);
  team_any<16>(A, u, b.head + (unsigned long long)u.part * 512 + lane * 16, b.end, parts, stack);
  if (u.part + 1 == u.k.upm && b.end - b.head != u.k.nbytes) {
    __syncthreads();   // the parts have been read
    if (sweep_dtype(u.k.meta) == HICCL_BF16) team_any<2>(A, u, edge_of<2>(u.k, b, lane), u.k.nbytes, parts, stack);
    else team_any<4>(A, u, edge_of<4>(u.k, b, lane), u.k.nbytes, parts, stack);
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
  if (v == 8) fold_any<W, 8, 4>(A, k, P, off, k.nbytes, stack, blockDim.x);
  else if (v == 2) fold_any<W, 2, 8>(A, k, P, off, k.nbytes, stack, blockDim.x);
  else fold_any<W, 1, 16>(A, k, P, off, k.nbytes, stack, blockDim.x);
}
template <bool ONE>
__global__ void SWEEP_BOUNDS(SWEEP_NARROW, 10) sweep_narrow_kernel(const __grid_constant__ SweepArgs A) {
  extern __shared__ uint32_t saved[];
  launch_order();
  each_unit<false>(A, [&](uint32_t unit) {
    const int lane = threadIdx.x & 31;
    const Unit u = find_unit(A, unit);
    if (sweep_lw(u.k.meta) == 2) narrow_unit<4>(A, u.k, u.P, u.part, lane, saved + threadIdx.x);
    else narrow_unit<2>(A, u.k, u.P, u.part, lane, saved + threadIdx.x);
  });
}

// Copies between operands that lie differently off a 16-byte boundary.  The
// source is read by its aligned vectors; the 16 bytes that a destination's
// vector takes straddle two of them, the lane's own and the next lane's, and
// are shifted out of the pair.  (Element accesses are bound by latency: 64
// bytes a warp request, 90 us for an odd-length BF16 All-to-all of 64 ranks x
// 1 MiB at four requests in flight and 45 us at sixteen, against 25 us here,
// 5.4 TB/s; aligned, it takes 23 us.  Two vectors a lane 27.2, eight 25.9 us.)  A unit is V rows of 31 destination vectors
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
__device__ __forceinline__ void shift_unit(const Unit &u, int lane) {
  const SweepClass &k = u.k;
  const unsigned long long *P = u.P;
  const uint32_t part = u.part;
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
  for (uint32_t d = u.d0; d < u.d1; ++d) {
    const unsigned long long dst = __ldg(P + d);
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
template <bool ONE>
__global__ void SWEEP_BOUNDS(SWEEP_SHIFT, 8) sweep_shift_kernel(const __grid_constant__ SweepArgs A) {
  launch_order();
  each_unit<ONE>(A, [&](uint32_t unit) {
    const Unit u = find_unit(A, unit);
    if (sweep_v(u.k.meta) == 4) shift_unit<4>(u, threadIdx.x & 31);
    else shift_unit<1>(u, threadIdx.x & 31);
  });
}

// ---- FP8 blocks --------------------------------------------------------------------
// A group of 8 lanes folds one 144-byte block, lane `sub` owning codes
// 16 * sub .. 16 * sub + 15; four blocks a warp.

struct Fp8Raw {
  uint4 c;
  float scale;
};

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

constexpr int FP8_GROUPS = 2;                                   // of the ring of an FP8 fold
constexpr uint32_t FP8_SLOTS = FP8_GROUPS * RING_GROUP;
constexpr uint32_t FP8_STEP = 4 * FP8_BLOCK_BYTES;              // bytes of a source in one slot

// blocks in shared memory: this lane's 16 codes (and the scale) of its group's
__device__ __forceinline__ Fp8Raw fp8_read(const char *block) {
  Fp8Raw x;
  x.c = *reinterpret_cast<const uint4 *>(block + 16 * (threadIdx.x & 7));
  x.scale = *reinterpret_cast<const float *>(block + 128);
  return x;
}
__device__ __forceinline__ void fp8_write(char *block, const Fp8Raw &r) {
  const uint32_t sub = threadIdx.x & 7;
  *reinterpret_cast<uint4 *>(block + 16 * sub) = r.c;
  if (sub == 0) *reinterpret_cast<uint4 *>(block + 128) = make_uint4(__float_as_uint(r.scale), 0u, 0u, 0u);
}
// A unit is four blocks, 576 bytes of every operand.  A source takes about 100
// instructions, so a warp is busy while its loads should fly; they pass
// through a ring of slots in shared memory, an asynchronous copy group for
// every RING_GROUP sources, which keeps loads in flight through folds,
// encodings and stores without holding registers (72 a thread, 24 warps an
// SM).  Copies and stores move the unit as one range of whole sectors, and
// only the fold reads it by blocks.  All-reduce of 16 Mi values a rank over 32 ranks ({4, 8}),
// 1.21 GB in and out: 265 us with the next sources loaded into registers (16
// warps an SM; 403 us when refilled one by one), 223 us through the ring by
// blocks, 199 us by the unit's range, 186 us (6.5 TB/s) with copy groups of
// four sources; two or four units a warp lose 5 and 10 %, neighbouring warps
// on neighbouring units read longer stretches of each source at a time.
struct Fp8Ring {
  const unsigned long long *P;
  uint32_t nsrc, lq, g, slot, ring_at;
  const char *mine;              // this lane's block in slot 0
  unsigned long long off;        // this lane's 16 bytes of the unit
  bool on, on2;                  // ... lie in the member; and 512 bytes further on (lanes 0 .. 3)

  __device__ __forceinline__ void load(uint32_t to_group) {
#pragma unroll
    for (uint32_t i = 0; i < RING_GROUP; ++i)
      if (lq + i < nsrc) {
        const unsigned long long s = pointer_at(P, lq + i, nsrc, held) + off;
        const uint32_t to = ring_at + (to_group * RING_GROUP + i) * FP8_STEP;
        if (on) cp_async16(to, s);
        if (on2) cp_async16(to + 512, s + 512);
      }
    lq += RING_GROUP;
    cp_commit();
  }
  __device__ __forceinline__ void start(const unsigned long long *sources, uint32_t n) {
    P = sources;
    nsrc = n;
    lq = g = 0;
#pragma unroll 1
    for (uint32_t i = 0; i < FP8_GROUPS - 1; ++i) load(i);
  }
  __device__ __forceinline__ Fp8Raw next(uint32_t q) {   // q = 0, 1, ...
    if (q % RING_GROUP == 0) {
      cp_wait<FP8_GROUPS - 2>();
      __syncwarp();              // every lane's copies have landed, and the group read last is free
      load(g == 0 ? FP8_GROUPS - 1 : g - 1);
      slot = g * RING_GROUP;
      if (++g == FP8_GROUPS) g = 0;
    }
    const Fp8Raw x = fp8_read(mine + slot * FP8_STEP);
    ++slot;
    return x;
  }
  __device__ __forceinline__ void drain() {              // the ring is free afterwards
    cp_wait<0>();
    __syncwarp();
  }

 private:
  unsigned long long held;
};

// the value of an expression, next(q) giving source q
template <typename NEXT>
__device__ __forceinline__ void fp8_fold(NEXT next, const uint32_t *tok, uint32_t nsrc, unsigned long long minus0,
                                         ulonglong2 *stack, uint32_t threads, unsigned long long (&acc)[8]) {
  uint32_t sp = 0;   // saved values end here
  Tokens t;
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] = 0ull;
#pragma unroll 1
  for (uint32_t q = 0; q < nsrc; ++q) {
    if ((q & 31u) == 0) t.read(tok, q, nsrc);
    unsigned long long y[8];
    fp8_widen(next(q), minus0, y);
    if (t.plain(q)) {
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i] = add2(acc[i], y[i]);
      continue;
    }
    const uint32_t tk = t.at(q);
    if (tk & TOK_START) {
      if (tk & TOK_PUSH) {
#pragma unroll
        for (int i = 0; i < 8; i += 2, sp += threads) stack[sp] = make_ulonglong2(acc[i], acc[i + 1]);
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
        sp -= 4 * threads;
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
          const ulonglong2 z = stack[sp + i / 2 * threads];
          acc[i] = add2(z.x, acc[i]);
          acc[i + 1] = add2(z.y, acc[i + 1]);
        }
      }
    }
  }
}

// the unit in slot 0 of the ring, as one range, to destinations d0, d0 + step, ...
__device__ __forceinline__ void fp8_store(const Unit &u, const Fp8Ring &ring, const char *slot0, uint32_t d0,
                                          uint32_t step) {
  const uint32_t lane = threadIdx.x & 31;
  __syncwarp();
  const uint4 v = *reinterpret_cast<const uint4 *>(slot0 + 16 * lane);
  const uint4 v2 = *reinterpret_cast<const uint4 *>(slot0 + 512 + 16 * (lane & 3));
#pragma unroll 4
  for (uint32_t d = d0; d < u.k.ndst; d += step) {
    const unsigned long long a = __ldg(u.P + u.k.nsrc + d) + ring.off;
    if (ring.on) *reinterpret_cast<uint4 *>(a) = v;
    if (ring.on2) *reinterpret_cast<uint4 *>(a + 512) = v2;
  }
}
__device__ __forceinline__ void fp8_ring_at(Fp8Ring &r, const Unit &u, char *base) {
  const uint32_t lane = threadIdx.x & 31;
  r.ring_at = static_cast<uint32_t>(__cvta_generic_to_shared(base)) + 16 * lane;
  r.mine = base + (lane >> 3) * FP8_BLOCK_BYTES;
  r.off = (unsigned long long)u.part * FP8_STEP + 16 * lane;
  r.on = r.off < u.k.nbytes;
  r.on2 = lane < 4 && r.off + 512 < u.k.nbytes;
}

template <bool ONE>
__global__ void SWEEP_BOUNDS(SWEEP_FP8, 6) sweep_fp8_kernel(const __grid_constant__ SweepArgs A) {
  extern __shared__ __align__(16) uint32_t saved[];
  launch_order();
  each_unit<ONE>(A, [&](uint32_t unit) {
    const Unit u = find_unit(A, unit);
    char *base = reinterpret_cast<char *>(saved) + (threadIdx.x >> 5) * (FP8_SLOTS * FP8_STEP);
    ulonglong2 *stack = reinterpret_cast<ulonglong2 *>(saved) + (blockDim.x >> 5) * (FP8_SLOTS * FP8_STEP / 16) + threadIdx.x;
    Fp8Ring ring;
    fp8_ring_at(ring, u, base);
    ring.start(u.P, u.k.nsrc);
    unsigned long long acc[8];
    fp8_fold([&](uint32_t q) { return ring.next(q); }, A.toks + u.k.tok, u.k.nsrc, A.minus0, stack, blockDim.x, acc);
    const Fp8Raw r = fp8_encode(acc);
    ring.drain();
    fp8_write(const_cast<char *>(ring.mine), r);
    fp8_store(u, ring, base, 0, 1);
    if constexpr (ONE) __syncwarp();   // slot 0 has been read
  });
}

// a short pass: a CTA to a unit, as sweep_team_kernel
template <bool MANY>
__global__ void __launch_bounds__(SWEEP_THREADS[SWEEP_FP8_TEAM], 2)
    sweep_fp8_team_kernel(const __grid_constant__ SweepArgs A) {
  __shared__ __align__(16) char few[MANY ? 16 : SWEEP_TEAM_STATIC * FP8_STEP];
  extern __shared__ __align__(16) uint32_t saved[];
  launch_order();
  const Unit u = find_unit(A, blockIdx.x);
  const SweepClass &k = u.k;
  char *parts = MANY ? reinterpret_cast<char *>(saved) : few;
  const uint32_t warp = threadIdx.x >> 5, warps = blockDim.x >> 5, grp = (threadIdx.x & 31) >> 3;
  char *rings = reinterpret_cast<char *>(saved) + (MANY ? A.sections * FP8_STEP : 0);
  char *base = rings + warp * (FP8_SLOTS * FP8_STEP);
  ulonglong2 *stack = reinterpret_cast<ulonglong2 *>(rings + warps * (FP8_SLOTS * FP8_STEP)) + threadIdx.x;
  const uint32_t *tok = A.toks + k.ttok, *bounds = tok + k.nsrc, *upper = bounds + k.team + 1;
  Fp8Ring ring;
  fp8_ring_at(ring, u, base);
  unsigned long long acc[8];
  for (uint32_t s = warp; s < k.team; s += warps) {
    const uint32_t q0 = __ldg(bounds + s), n = __ldg(bounds + s + 1) - q0;
    ring.start(u.P + q0, n);
    Fp8Raw only;   // a section of one source passes its block through
    fp8_fold([&](uint32_t q) { return only = ring.next(q); }, tok + q0, n, A.minus0, stack, blockDim.x, acc);
    const Fp8Raw r = fp8_encode(acc);
    fp8_write(parts + s * FP8_STEP + grp * FP8_BLOCK_BYTES, n == 1 ? only : r);
    ring.drain();
  }
  __syncthreads();
  fp8_fold([&](uint32_t s) { return fp8_read(parts + s * FP8_STEP + grp * FP8_BLOCK_BYTES); }, upper, k.team, A.minus0,
           stack, blockDim.x, acc);
  fp8_write(const_cast<char *>(ring.mine), fp8_encode(acc));
  fp8_store(u, ring, base, warp, warps);
}

}  // namespace

}  // namespace hiccl
