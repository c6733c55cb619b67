// Streamed operators of the AMG-preconditioned Krylov solvers, prefetched through shared memory.
//
// A solve applies the same operators in the same order every iteration (the V-cycle's level
// operators, then the matrix), each warp always the same contiguous share of each of them, and
// the operators never change during a solve.  Only the gathered vectors depend on earlier phases.
// So every warp keeps a ring of kSlots slots of kSlotBytes in shared memory and fetches the
// elements (column, value) of its shares ahead of their use with bulk asynchronous copies
// (cp.async.bulk), running through the phases in their cyclic order and across the barriers
// between them: when a phase starts, its first elements are already on chip, and the memory
// system stays busy while the blocks wait for each other.  What is left on a phase's critical
// path is one gather, the row's epilogue and the barrier.
//
// Bulk copies complete on an mbarrier and belong to the async proxy, so the release fence of a
// barrier does not wait for them; with cp.async it did (1,350 -> 2,330 cycles for a cluster barrier
// of 16 x 512 threads with one 16-byte copy per thread in flight, more under load).
//
// A slot holds a fixed number of 32-element steps of one phase (steps_per_slot).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "avip_internal.h"
#include "sell.cuh"

namespace avip {

constexpr int kSlotBytes = 2048;
constexpr int kMaxPhases = 2 * kAmgMaxLevels;  // 2 nlev - 1 of the V-cycle, and the matrix
static_assert(kMaxPhases <= 32, "one lane per phase");

__device__ __forceinline__ void mbar_init(uint32_t bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t bar, int bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// The elements are read once per product: evict-first, so that they do not push the gathered
// vectors out of L2 (500,000 rows: without the policy a solve wrote 588 MB of vectors back to DRAM).
__device__ __forceinline__ unsigned long long evict_first_policy() {
  unsigned long long p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, int bytes, uint32_t bar,
                                          unsigned long long policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
          dst),
      "l"(src), "r"(bytes), "r"(bar), "l"(policy)
      : "memory");
}
// Bound of every wait for a copy (each try suspends the warp for up to a hardware time limit).
constexpr int kCopyTries = 1 << 20;

// One phase's operator: a SELL-32 matrix whose columns carry bit 31 on the last step of every
// slice, or, with col == nullptr, a dense row-major matrix with rows padded to whole steps.
struct PhaseDesc {
  const int32_t* col;
  const void* val;
  const int32_t* sl_ptr;  // first element of each slice (sparse)
  int32_t nslices;        // slices (sparse) or rows (dense)
  int32_t nrows;
  int32_t lpr;            // lanes per row (sparse) or steps per row (dense)
  int32_t wide;           // 1: 8-byte values
};

// Steps of 32 elements per slot.
template <typename TV, bool kDense>
__host__ __device__ constexpr int steps_per_slot() {
  return kDense ? kSlotBytes / (32 * (int)sizeof(TV)) : (sizeof(TV) == 4 ? 8 : 4);
}

// One warp's ring and its shares: lane p holds the share of phase p.
template <int kSlots>
struct Ring {
  static_assert(kSlots <= 8, "bits of state");
  static constexpr int kDepth = kSlots;
  static constexpr unsigned kAll = (1u << kSlots) - 1u;
  static constexpr int kWarpBytes = kSlots * kSlotBytes;
  const PhaseDesc* tab;  // shared memory
  char* buf;             // this warp's slots
  uint32_t sbuf, bar;    // shared addresses of the slots and of their mbarriers
  int e0, ns, sa;        // lane p: first element, steps and first slice (row) of this warp in phase p
  unsigned live;         // phases in which this warp has steps
  int cph;               // phase whose first step the oldest slot holds
  int slot;              // oldest slot
  unsigned state;        // bit k: parity of slot k's current fetch; bit 31: this lane gave up a wait; bit 30: the warp
                         // has, bits 8 + k then: slot k has a copy in flight
  int pph, prem;         // next phase to fetch from and its steps left
  const char *pcol, *pval;
  int rs;                // lane p: first slot of phase p when everything stays resident
  bool resident;         // the warp's shares of all phases fit its slots: fetched once per solve
  unsigned long long policy;
  volatile int* bad;     // shared memory: set when a wait for a copy is given up

  __device__ __forceinline__ int next_live(int ph) const {
    const unsigned above = live & ~((2u << ph) - 1u);
    return __ffs(above ? above : live) - 1;
  }
  __device__ __forceinline__ void point(int ph) {
    pph = ph;
    prem = __shfl_sync(0xffffffffu, ns, ph);
    const size_t e = (size_t)(unsigned)__shfl_sync(0xffffffffu, e0, ph);
    const PhaseDesc& d = tab[ph];
    pcol = reinterpret_cast<const char*>(d.col) + e * 4;
    pval = static_cast<const char*>(d.val) + (e << (d.wide ? 3 : 2));
  }
  // Fetch the next steps into slot k (only called with live != 0).  A slot is always filled: past
  // the end of the warp's share come the next rows' elements (or the arrays' padding), which
  // stream_rows gathers for but never emits, so its steps need no predicates.
  __device__ __forceinline__ void issue(int k, int lane) {
    const PhaseDesc& d = tab[pph];
    const bool dense = d.col == nullptr, wide = d.wide != 0;
    const int cap = dense ? (wide ? 8 : 16) : (wide ? 4 : 8);
    const int vbytes = cap << (wide ? 8 : 7), cbytes = dense ? 0 : cap << 7;
    if (lane == 0) {
      const uint32_t s = sbuf + k * kSlotBytes, b = bar + k * 8;
      mbar_expect(b, vbytes + cbytes);
      if (!dense) bulk_copy(s, pcol, cbytes, b, policy);
      bulk_copy(s + cbytes, pval, vbytes, b, policy);
    }
    pcol += cbytes;
    pval += vbytes;
    prem -= cap;
    if (prem <= 0) point(next_live(pph));
  }
  __device__ __forceinline__ bool given_up() const { return state >> 30 & 1u; }
  // Mask of a slot's columns: without the end-of-slice bit; 0 on a lane that gave up.
  __device__ __forceinline__ int column_mask() const { return ~((int)state >> 31) & 0x7fffffff; }
  __device__ __forceinline__ bool arrived(int k) const { return mbar_try(bar + k * 8, (state >> k) & 1u); }
  // Wait for slot k's fetch.  A lane that gives up, or sees that another warp of the block has, goes on
  // with columns of 0 (a stale one would gather from anywhere); the warp agrees on it where it has to
  // meet anyway, before it refills the slot (advance: a vote here costs 0.4 to 0.8 % of a solve).
  __device__ __forceinline__ void wait(int k) {
    if (!arrived(k)) {
      int t = 0;
      while (!arrived(k))
        if (*bad || ++t == kCopyTries) {
          *bad = 1;
          state |= 1u << 31;
          return;
        }
    }
    state ^= 1u << k;
  }
  // (all lanes) No steps any more: the slots of `flying` keep their copies in flight for finish(), and the
  // solve leaves at its next sum or grid barrier, which look at *bad.
  __device__ __forceinline__ void give_up(unsigned flying) {
    if (!given_up()) state |= 1u << 30 | flying << 8;
    ns = 0;
    *bad = 1;
  }
  // Drop what was fetched and fetch from the start of phase ph on.
  __device__ __forceinline__ void restart(int ph, int lane) {
    drain();
    slot = 0;
    cph = ph;
    if (given_up()) return;
    point(ph);
#pragma unroll 1
    for (int k = 0; k < kSlots; ++k) issue(k, lane);
  }
  // This warp's shares of the n phases of `t` (shared memory, complete); the first fetches
  // start at phase `first`.  `b`: this warp's slots, `mb`: its kSlots mbarriers; no_wait: give up the
  // first wait (the failure path's test).
  __device__ __forceinline__ void init(const PhaseDesc* t, int n, char* b, unsigned long long* mb, int* bad_flag, int gwarp,
                                       int nwarps, int lane, int first, bool no_wait) {
    tab = t;
    buf = b;
    sbuf = (uint32_t)__cvta_generic_to_shared(b);
    bar = (uint32_t)__cvta_generic_to_shared(mb);
    bad = bad_flag;
    policy = evict_first_policy();
    state = 0;
    if (lane < kSlots) mbar_init(bar + lane * 8);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    e0 = ns = sa = 0;
    if (lane < n) {
      const PhaseDesc& d = t[lane];
      int sb;
      warp_slices(d.nslices, gwarp, nwarps, sa, sb);
      if (sb > sa) {
        if (d.col) {
          e0 = __ldg(d.sl_ptr + sa);
          ns = (__ldg(d.sl_ptr + sb) - e0) >> 5;
        } else {
          e0 = sa * d.lpr * 32;
          ns = (sb - sa) * d.lpr;
        }
      }
    }
    live = __ballot_sync(0xffffffffu, ns > 0);
    cph = -1;
    slot = 0;
    // slots of each phase, and their prefix sum in phase order
    int need = 0;
    if (ns > 0) {
      const PhaseDesc& d = t[lane];
      const int cap = d.col ? (d.wide ? 4 : 8) : (d.wide ? 8 : 16);
      need = (ns + cap - 1) / cap;
    }
    rs = need;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, rs, o);
      if (lane >= o) rs += v;
    }
    const int total = __shfl_sync(0xffffffffu, rs, 31);
    rs -= need;
    resident = total <= kSlots;
    if (live) {
      cph = resident ? __ffs(live) - 1 : ((live >> first) & 1u) ? first : next_live(first);
      point(cph);
      const int n0 = resident ? total : kSlots;
#pragma unroll 1
      for (int k = 0; k < n0; ++k) issue(k, lane);
      if (no_wait) {
        give_up((1u << n0) - 1u);
      } else if (resident) {
#pragma unroll 1
        for (int k = 0; k < n0; ++k) {
          wait(k);
          if (!agree(k, (1u << n0) - (1u << k))) break;
        }
      }
    }
  }
  // First slot of phase ph's next steps, and the step after a slot has been used.
  __device__ __forceinline__ int enter(int ph, int lane) {
    if (resident) return __shfl_sync(0xffffffffu, rs, ph);
    if (cph != ph) restart(ph, lane);
    return slot;
  }
  __device__ __forceinline__ bool agree(int k, unsigned flying) {
    if (__all_sync(0xffffffffu, (int)state >= 0)) return true;
    if ((int)state >= 0) state ^= 1u << k;
    give_up(flying);
    return false;
  }
  // False (on all lanes) when a lane gave up the wait for slot k.
  __device__ __forceinline__ bool advance(int& k, int lane) {
    if (resident) {
      ++k;
      return true;
    }
    if (!agree(k, kAll)) return false;
    issue(k, lane);
    k = slot = k + 1 == kSlots ? 0 : k + 1;
    return true;
  }
  __device__ __forceinline__ void leave(int ph) {
    if (!resident) cph = next_live(ph);
  }
  // Wait for every copy in flight, whatever was given up: none may be when the slots are given back or
  // refilled out of order.
  __device__ __forceinline__ void drain() {
    const unsigned flying = given_up() ? state >> 8 & kAll : live && !resident ? kAll : 0u;
    state &= ~(kAll << 8);
#pragma unroll 1
    for (int k = 0; k < kSlots; ++k)
      if (flying >> k & 1u) {
        int t = 0;
        while (!__all_sync(0xffffffffu, arrived(k)))
          if (++t == kCopyTries) {
            give_up(0u);
            break;
          }
        state ^= 1u << k;
      }
    __syncwarp();
  }
  // End of a solve: nothing in flight, and the mbarriers may be initialised again.
  __device__ __forceinline__ void finish(int lane) {
    drain();
    if (lane < kSlots) asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(bar + lane * 8) : "memory");
    __syncwarp();
  }
};

// No operands to fetch ahead for a row.
struct NoPre {};
struct NoBegin {
  __device__ NoPre operator()(int) const { return NoPre(); }
};

// This warp's rows of the sparse operator of phase ph: emit(row, sum of val * g(col), pre) for
// every row, in slice order, on the row's first lane, with pre = begin(row) evaluated when the
// row's slice starts so that its loads overlap the slice's gathers.  Padding elements (column 0,
// value 0) are read like the others and add nothing.  The lanes of a row combine their sums by
// shuffles at the slice's last step (bit 31 of the column, the same on all 32 lanes).  The
// epilogue stands once in the code, in a loop over the slot's slice ends, and not in every
// unrolled step: a phase of a small mesh runs through its code once, and is then bound by
// instruction fetch and issue latency.
template <typename TA, typename TV, class R, class G, class Begin, class Emit>
__device__ __forceinline__ void stream_rows(R& ring, int ph, int lane, G g, Begin begin, Emit emit) {
  const int nsteps = __shfl_sync(0xffffffffu, ring.ns, ph);
  if (nsteps == 0) return;
  int k = ring.enter(ph, lane);
  constexpr int K = steps_per_slot<TV, false>();
  const PhaseDesc& d = ring.tab[ph];
  const int nrows = d.nrows, lpr = d.lpr, lg = __ffs(lpr) - 1;
  const bool lead = (lane & (lpr - 1)) == 0;
  int row = (__shfl_sync(0xffffffffu, ring.sa, ph) << (5 - lg)) + (lane >> lg);
  decltype(begin(0)) pre{};
  if (lead && row < nrows) pre = begin(row);
  TA acc = TA(0);
#pragma unroll 1
  for (int left = nsteps; left > 0; left -= K) {
    if (!ring.resident) ring.wait(k);
    const char* s = ring.buf + k * kSlotBytes;
    const int32_t* cs = reinterpret_cast<const int32_t*>(s) + lane;
    const TV* vs = reinterpret_cast<const TV*>(s + K * 128) + lane;
    const int cmask = ring.column_mask();
    TA x[K], v[K];
#pragma unroll
    for (int u = 0; u < K; ++u) x[u] = (TA)g(cs[u * 32] & cmask);
    // bit u: step u ends a slice (lane u looks at step u)
    unsigned ends = __ballot_sync(0xffffffffu, lane < K && lane < left && cs[lane * 32 - lane] < 0);
#pragma unroll
    for (int u = 0; u < K; ++u) v[u] = vs[u * 32];
    unsigned todo = (1u << K) - 1u;
    while (true) {
      const unsigned seg = ends ? todo & ((2u << (__ffs(ends) - 1)) - 1u) : todo;
#pragma unroll
      for (int u = 0; u < K; ++u)
        if (seg >> u & 1u) acc = fma_t(v[u], x[u], acc);
      if (!ends) break;
      todo &= ~seg;
      ends &= ends - 1u;
      for (int o = lpr >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lead && row < nrows) emit(row, acc, pre);
      acc = TA(0);
      row += 32 >> lg;
      if (lead && row < nrows && (ends || left > K)) pre = begin(row);
      if (!ends && left <= K) break;
    }
    if (!ring.advance(k, lane)) return;
  }
  ring.leave(ph);
}

// This warp's rows of the dense operator of phase ph: out(row, sum_k M[row, k] b[k], pre) on lane 0, b
// (the whole right-hand side) in shared memory, pre = begin(row) evaluated when the row starts.  Rows
// of at least a slot (the inverses of small matrices, the V-cycle's tail) take the slot's steps of
// one row at a time, all loads before the sums; with a test of the row's end after every step the
// loads of a step waited for the sums of the last one (65 x 65 nodes, 71 MB over the GPU: 75.4 ->
// 65.4 us per solve of 1.34 iterations; 500,000 nodes, tail of 1,073 rows: 77.9 -> 76.4 us per
// iteration).  Shorter rows, of which a slot holds several, keep that form.
template <typename T, class R, class Begin, class Out>
__device__ __forceinline__ void stream_dense(R& ring, int ph, int lane, const T* b, Begin begin, Out out) {
  const int nsteps = __shfl_sync(0xffffffffu, ring.ns, ph);
  if (nsteps == 0) return;
  int slot = ring.enter(ph, lane);
  constexpr int K = steps_per_slot<T, true>();
  const int w = ring.tab[ph].lpr, nrows = ring.tab[ph].nslices;
  int row = __shfl_sync(0xffffffffu, ring.sa, ph), k = 0;
  T acc = T(0);
  decltype(begin(0)) pre{};
  if (lane == 0) pre = begin(row);
  auto end_row = [&]() {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) {
      out(row, acc, pre);
      if (row + 1 < nrows) pre = begin(row + 1);
    }
    acc = T(0);
    k = 0;
    ++row;
  };
#pragma unroll 1
  for (int left = nsteps; left > 0; left -= K) {
    if (!ring.resident) ring.wait(slot);
    const T* vs = reinterpret_cast<const T*>(ring.buf + slot * kSlotBytes) + lane;
    const int cnt = min(K, left);
    if (w >= K) {
#pragma unroll 1
      for (int u = 0; u < cnt;) {
        const int n = min(cnt - u, w - k);
        const T *vp = vs + u * 32, *bp = b + k * 32 + lane;
        if (n == K) {
          T v[K], x[K];
#pragma unroll
          for (int q = 0; q < K; ++q) {
            v[q] = vp[q * 32];
            x[q] = bp[q * 32];
          }
#pragma unroll
          for (int q = 0; q < K; ++q) acc = fma_t(v[q], x[q], acc);
        } else {
#pragma unroll 4
          for (int q = 0; q < n; ++q) acc = fma_t(vp[q * 32], bp[q * 32], acc);
        }
        u += n;
        k += n;
        if (k == w) end_row();
      }
    } else {
#pragma unroll 4
      for (int u = 0; u < cnt; ++u) {
        acc = fma_t(vs[u * 32], b[k * 32 + lane], acc);
        if (++k == w) end_row();
      }
    }
    if (!ring.advance(slot, lane)) return;
  }
  ring.leave(ph);
}

}  // namespace avip
