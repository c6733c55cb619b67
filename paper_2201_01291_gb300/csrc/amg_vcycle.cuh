// Smoothed-aggregation AMG V-cycle shared by the whole-GPU cooperative solvers (grid-wide
// barriers) and the cluster solvers (one thread-block cluster per instance, cluster barriers).
//
// Each non-coarsest level takes two phases, through the composite operators built on the host
// (amg_setup.cpp): down, xp = Q b and b' = Rf b (the pre-smoothing, the residual and its
// restriction); up, x = U xp + Pf x' (the coarse correction and the post-smoothing).  It is the
// V-cycle of a damped Jacobi smoother (the same step before and after), R = P^T and a dense
// coarsest solve, written with fewer grid-wide phases: every phase gathers only vectors
// completed by an earlier one.  The values are FP32 by default (the preconditioner only shapes
// the search directions; the iterate, the residuals and the stopping test stay FP64) or FP64.
//
// The levels below the finest one of at most kAmgDenseRows rows are applied as one dense product
// (AmgDenseT): phase p of the cycle is the down phase of level p for p < dl (the dense level), the
// dense product for p = dl, the up phase of level 2 dl - p above, and phase 2 dl + 1 is the
// product with the matrix.  Every operator streams through the warps' rings (stream.cuh).
//
// `Ops` supplies the synchronisation of the participating threads: barrier() completes every
// vector written before it, sum(v) returns the sum of v over all participants (and is a
// barrier too); both return false if a wait was abandoned.  ops.ring is the calling warp's ring,
// gwarp / nwarps number the participating warps.
#pragma once
#include <cooperative_groups.h>

#include <type_traits>

#include "avip_internal.h"
#include "grid_sync.cuh"
#include "sell.cuh"
#include "stream.cuh"

namespace avip {

// Per-thread accumulation of a dot product: FP64 fused multiply-adds, or compensated (Kahan)
// FP32 sums in the mixed-precision solve.
template <typename T>
struct DotAcc;
template <>
struct DotAcc<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double a, double b) { s = fma(a, b, s); }
  __device__ __forceinline__ double value() const { return s; }
};
template <>
struct DotAcc<float> {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float a, float b) {
    const float y = a * b - c;
    const float t = s + y;
    c = (t - s) - y;
    s = t;
  }
  __device__ __forceinline__ double value() const { return (double)s - (double)c; }
};

// A solve's hierarchy and phase table in shared memory (one per block), and its dense level.
struct SolveShared {
  PhaseDesc tab[kMaxPhases];
  unsigned long long H[sizeof(AmgDevT<double>) / 8];
  unsigned long long bar[128];      // the rings' mbarriers, kDepth per warp
  double gain;
  int bad;                          // a warp gave up the wait for a copy (Ring::wait)
};
// Dynamic shared memory of a solve: the rings, then the dense product's right-hand side.
constexpr size_t kRhsBytes = sizeof(float) * kInverseRows;
static_assert(kRhsBytes >= sizeof(double) * kAmgDenseRows, "an FP64 hierarchy has no inverse of the finest matrix");
template <typename T>
struct AmgCtx {
  const AmgDevT<T>* H;  // shared memory
  AmgDenseT<T> D;
  double gain;          // of the Dirichlet lift (dirichlet_gain; a division, so one thread per block)
  T* rhs;               // shared memory: the dense product's right-hand side, zero-padded
  __device__ __forceinline__ int mat_phase() const { return 2 * D.level + 1; }
};

// The finest dense operator whose share per CTA and product stays within a bound: kInverseBytesPerCta
// for the inverse of the matrix, kDenseBytesPerCta for the V-cycle's tail; the coarsest inverse on
// fewer CTAs.
template <typename T>
__device__ __forceinline__ int dense_choice(const AmgDevT<T>& H, int nctas) {
  auto bytes = [&](int k) {
    return (size_t)H.L[H.dense[k].level].n * H.dense[k].steps * kSlice * sizeof(T);
  };
  if (H.dense[0].m && bytes(0) <= kInverseBytesPerCta * (size_t)nctas) return 0;
  return bytes(1) <= kDenseBytesPerCta * (size_t)nctas ? 1 : 2;
}

// Start of a solve: the hierarchy's descriptors copied to shared memory, the phase table written
// and the calling warp's ring started at the matrix phase (the solve begins with a true residual)
// or at the finest down phase.  TA: type of the streamed matrix values.  Every thread of the
// participating blocks calls it.
// keep: the dense operator is the coarsest inverse whatever the number of CTAs (the mixed-precision
// solves' arithmetic, see block_group_sum).
template <typename T, typename TA, class R>
__device__ AmgCtx<T> solve_begin(SolveShared& sh, R& ring, char* dyn, const PcgArgs& a,
                                 const AmgDevT<T>* __restrict__ Hg, const TA* aval, int nctas, int gwarp, int nwarps,
                                 int lane, bool matrix_first, bool keep = false) {
  static_assert(sizeof(AmgDevT<T>) == sizeof(AmgDevT<double>), "one shared copy for both types");
  const unsigned long long* src = reinterpret_cast<const unsigned long long*>(Hg);
  for (int k = threadIdx.x; k < (int)(sizeof(AmgDevT<T>) / 8); k += blockDim.x) sh.H[k] = src[k];
  if (threadIdx.x == 0) {
    sh.gain = dirichlet_gain(a);
    sh.bad = 0;
  }
  __syncthreads();
  AmgCtx<T> C;
  C.gain = sh.gain;
  C.rhs = reinterpret_cast<T*>(dyn + (blockDim.x >> 5) * R::kWarpBytes);
  C.H = reinterpret_cast<const AmgDevT<T>*>(sh.H);
  C.D = C.H->dense[keep ? 2 : dense_choice(*C.H, nctas)];
  const int dl = C.D.level, p = (int)threadIdx.x;
  if (p <= 2 * dl + 1) {
    PhaseDesc d;
    if (p == 2 * dl + 1) {
      d = PhaseDesc{a.colS, aval, a.A.sl_ptr, a.A.nslices, a.A.N, 1, sizeof(TA) == 8};
    } else if (p == dl) {
      const int n = C.H->L[dl].n;
      d = PhaseDesc{nullptr, C.D.m, nullptr, n, n, C.D.steps, sizeof(T) == 8};
    } else {
      const SellMatT<T>& M = p < dl ? C.H->L[p].Rf : C.H->L[2 * dl - p].UP;
      d = PhaseDesc{M.col, M.val, M.sl_ptr, M.nslices, M.n, M.lpr, sizeof(T) == 8};
    }
    sh.tab[p] = d;
  }
  __syncthreads();
  ring.init(sh.tab, 2 * dl + 2, dyn + (threadIdx.x >> 5) * R::kWarpBytes,
            sh.bar + (threadIdx.x >> 5) * R::kDepth, &sh.bad, gwarp, nwarps, lane, matrix_first ? 2 * dl + 1 : 0,
            a.spin_ns == 0);
  return C;
}

// Down phase of level l: xp = Q b on the rows of level l (Q = omega D^-1 is diagonal: an
// elementwise pass) and b' = Rf b on the rows of level l + 1 (a streamed product), b given by
// `src` (complete on entry).  `hook` takes part in every row i of level l: hook.begin(i) loads
// the row's own operands, hook.end(i, pre) runs with them (the CG update folded into the
// finest level's phase).
template <typename T, class Ops, class Src, class Hook>
__device__ __forceinline__ void amg_down(const AmgCtx<T>& C, Ops& ops, int l, Src src, Hook hook, int gwarp,
                                         int nwarps, int lane) {
  const AmgLevelT<T>& L = C.H->L[l];
  T* __restrict__ bn = C.H->L[l + 1].b;
  T* __restrict__ xp = L.xp;
  const T* __restrict__ qd = L.qd;
  const int n = L.n;
  // two rows per thread at a time, their loads issued together
  const int stride = nwarps * kSlice;
  for (int i = gwarp * kSlice + lane; i < n; i += 2 * stride) {
    const int j = i + stride;
    const bool two = j < n;
    const auto pi = hook.begin(i);
    const T bi = src(i), qi = __ldg(qd + i);
    const auto pj = hook.begin(two ? j : i);
    const T bj = src(two ? j : i), qj = __ldg(qd + (two ? j : i));
    hook.end(i, pi);
    xp[i] = qi * bi;
    if (two) {
      hook.end(j, pj);
      xp[j] = qj * bj;
    }
  }
  stream_rows<T, T>(ops.ring, l, lane, src, NoBegin(), [&](int j, T v, NoPre) { bn[j] = v; });
}

// Up phase of level l: x = U xp + Pf x' = [U | Pf] [xp; x'] on the rows of level l (x' = the
// next level's solution, complete on entry), each row handed to out.end(i, value, pre) with the
// operands out.begin(i) fetched ahead.
template <typename T, class Ops, class Out>
__device__ __forceinline__ void amg_up(const AmgCtx<T>& C, Ops& ops, int l, Out out, int lane) {
  const AmgLevelT<T>& L = C.H->L[l];
  const T* __restrict__ xp = L.xp;  // followed by x'
  stream_rows<T, T>(ops.ring, 2 * C.D.level - l, lane, [xp](int c) { return __ldca(xp + c); },
                    [&](int i) { return out.begin(i); },
                    [&](int i, T v, const decltype(out.begin(0))& pre) { out.end(i, v, pre); });
}

// Row hooks and outputs without prefetched operands.
struct NoHook {
  __device__ NoPre begin(int) const { return NoPre(); }
  __device__ void end(int, NoPre) const {}
};
template <typename T>
struct StoreOut {  // x_i = value
  T* x;
  __device__ NoPre begin(int) const { return NoPre(); }
  __device__ void end(int i, T v, NoPre) const { x[i] = v; }
};

// The dense product x = M b of the phase dl, b given by src: every block first copies all of b to
// shared memory, so that the product's inner loop has no memory latency.
template <typename T, class Ops, class Src, class Out>
__device__ __forceinline__ void amg_dense(const AmgCtx<T>& C, Ops& ops, Src src, Out out, int lane) {
  const int n = C.H->L[C.D.level].n, np = C.D.steps * kSlice;
  for (int k0 = threadIdx.x; k0 < np; k0 += 4 * blockDim.x) {
    T v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int k = k0 + q * blockDim.x;
      v[q] = k < n ? src(k) : T(0);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int k = k0 + q * blockDim.x;
      if (k < np) C.rhs[k] = v[q];
    }
  }
  __syncthreads();
  using P = decltype(out.begin(0));
  stream_dense<T>(ops.ring, C.D.level, lane, C.rhs, [&out](int row) { return out.begin(row); },
                  [&out](int row, T v, P p) { out.end(row, v, p); });
}

// The V-cycle below the finest level: down phases of levels 1 .. dl-1, the dense product, up
// phases of levels dl-1 .. 1, one barrier after each.  Entered once the finest down phase is
// complete (dl >= 1); on return the level-1 solution is complete.
template <typename T, class Ops>
__device__ bool amg_inner(const AmgCtx<T>& C, Ops& ops, int gwarp, int nwarps, int lane) {
  const int dl = C.D.level;
  for (int l = 1; l < dl; ++l) {
    const T* __restrict__ b = C.H->L[l].b;
    amg_down(C, ops, l, [b](int c) { return __ldca(b + c); }, NoHook(), gwarp, nwarps, lane);
    if (!ops.barrier()) return false;
  }
  {
    const T* __restrict__ cb = C.H->L[dl].b;
    T* __restrict__ cx = C.H->L[dl].x;
    amg_dense(C, ops, [cb](int k) { return __ldca(cb + k); }, StoreOut<T>{cx}, lane);
    if (!ops.barrier()) return false;
  }
  for (int l = dl - 1; l >= 1; --l) {
    amg_up(C, ops, l, StoreOut<T>{C.H->L[l].x}, lane);
    if (!ops.barrier()) return false;
  }
  return true;
}

// One V-cycle z = M b0, b0 complete on entry (TB: its type; TZ: the type z is stored in).  With
// an epilogue (NE > 0) the last barrier is a sum of b0.z handed to it (sum_epi); otherwise a plain
// barrier.  Returns false if a wait was abandoned.
template <typename T, typename TB, typename TZ, class Ops, int NE, class Epi>
__device__ bool vcycle(const AmgCtx<T>& C, const TB* __restrict__ b0, TZ* __restrict__ z, Ops& ops, int gwarp,
                       int nwarps, int lane, double (&res)[NE], bool& flag, Epi epi) {
  constexpr bool kDot = !std::is_same<Epi, NoEpilogue>::value;
  auto src = [b0](int c) { return (T)__ldca(b0 + c); };
  DotAcc<double> acc;
  struct Out {  // z_i = value, b0_i z_i into the dot product
    const TB* b0;
    TZ* z;
    DotAcc<double>* acc;
    __device__ TB begin(int i) const { return kDot ? __ldca(b0 + i) : TB(0); }
    __device__ void end(int i, T v, TB bi) const {
      z[i] = (TZ)v;
      if (kDot) acc->add((double)bi, (double)v);
    }
  } out{b0, z, &acc};
  if (C.D.level == 0) {
    amg_dense(C, ops, src, out, lane);
  } else {
    amg_down(C, ops, 0, src, NoHook(), gwarp, nwarps, lane);
    if (!ops.barrier()) return false;
    if (!amg_inner(C, ops, gwarp, nwarps, lane)) return false;
    amg_up(C, ops, 0, out, lane);
  }
  if constexpr (kDot) {
    return ops.template sum_epi<NE>(acc.value(), res, flag, epi);
  } else {
    return ops.barrier();
  }
}
template <typename T, typename TB, typename TZ, class Ops>
__device__ bool vcycle(const AmgCtx<T>& C, const TB* __restrict__ b0, TZ* __restrict__ z, Ops& ops, int gwarp,
                       int nwarps, int lane) {
  double none[1];
  bool flag;
  return vcycle(C, b0, z, ops, gwarp, nwarps, lane, none, flag, NoEpilogue());
}

// CG preconditioned by the V-cycle on the scaled system (kinds 8, 11 and the batched FP64 form):
// warm start, b', true-residual checks and restarts, phi = D^-1/2 x.  The hierarchy H (values of
// type T) writes the preconditioned residual z in FP64 (only w = A z gathers it).  The residual update r - alpha q and
// x += alpha p of iteration k are folded into the finest down phase of iteration k + 1, whose
// products gather r - alpha q directly (the new residual goes to the other buffer, r2), so an
// iteration takes 2 dl + 2 grid-wide phases: the finest down phase (sum of r.r: stop test), the
// levels below, the finest up phase (sum of r.z), and w = A z (sum of p.q).  `leader` is the
// one thread that writes the solve statistics.  Returns false if a wait was abandoned.
template <typename T, class Ops>
__device__ bool amg_cg_solve(const PcgArgs& a, const AmgCtx<T>& C, double* __restrict__ z, Ops& ops, int gwarp,
                             int nwarps, int lane, bool leader) {
  constexpr int kMaxRestarts = 8;
  const int N = a.A.N, nsl = a.A.nslices, dl = C.D.level, mat = C.mat_phase();
  const double* nb = a.nbuf + (size_t)a.sc->parity * AVIP_MAX_SPECIES * a.Npad;

  // ---- x = D^1/2 phi (warm start) and b'
  const double gain = C.gain;
  const int hist = history_length(a);
  double bb[1] = {0.0};
  for (int s = gwarp; s < nsl; s += nwarps) {
    const int i = s * kSlice + lane;
    if (i >= N) continue;
    a.x[i] = a.dsq[i] * predict_phi(a, i, hist);
    double b;
    if (a.use_density_rhs) {
      double rho = 0.0;
      if (a.rhs_src)
        rho = a.rhs_src[i];
      else
        for (int k = 0; k < a.ns; ++k) rho = fma(a.q[k], nb[(size_t)k * a.Npad + i], rho);
      b = fma(a.rhs_scale[i], rho, gain * a.lift[i]);
      a.b[i] = b;
    } else {
      b = a.b[i];
    }
    if (a.rhs_scale[i] != 0.0) bb[0] = fma(b, b, bb[0]);  // free rows only: a Dirichlet row holds its value exactly
    else a.x[i] = b;  // a Dirichlet unit row takes its (possibly ramped) value exactly
  }
  if (!ops.sum(bb)) return false;
  {
    const double thresh = a.rtol * a.rtol * bb[0];
    double* rc = a.r;   // current residual
    double* rn = a.r2;  // the other buffer
    // the vectors the finest down phase gathers, in the hierarchy's type: with T = float, FP32
    // copies of r (both buffers) and q, written beside them; with T = double, r and q themselves
    constexpr bool kCopies = sizeof(T) == 4;
    T* tc = kCopies ? (T*)a.rq32 : (T*)rc;
    T* tn = kCopies ? (T*)a.rq32 + a.Npad : (T*)rn;
    T* tq = kCopies ? (T*)a.rq32 + 2 * (size_t)a.Npad : (T*)a.q_ap;
    double rz = 0.0, rr_true = 0.0, alpha = 0.0;
    bool check = true, fresh = true;
    int it = 0, restarts = 0, status = AVIP_OK;
    if (bb[0] == 0.0) {
      for (int s = gwarp; s < nsl; s += nwarps) {
        const int i = s * kSlice + lane;
        if (i < N) a.x[i] = a.b[i];  // free b == 0: x = b
      }
    } else {
      while (true) {
        if (check || it >= a.max_iter) {
          // ---- true residual r = b' - A x (x complete)
          double r2[1] = {0.0};
          {
            const double* __restrict__ xv = a.x;
            const double* __restrict__ bv = a.b;
            double* __restrict__ rw = rc;
            T* __restrict__ tw = tc;
            stream_rows<double, double>(
                ops.ring, mat, lane, [xv](int c) { return __ldca(xv + c); }, [bv](int i) { return bv[i]; },
                [&](int i, double ax, double bi) {
                  const double r = bi - ax;
                  rw[i] = r;
                  if (kCopies) tw[i] = (T)r;
                  r2[0] = fma(r, r, r2[0]);
                });
          }
          double tot[1];
          bool small;
          if (!ops.template sum_epi<1>(r2[0], tot, small, [thresh](double t, double* o) {
                o[0] = t;
                return t <= thresh;
              }))
            return false;
          rr_true = tot[0];
          if (small) break;
          if (!isfinite(rr_true)) {  // non-finite data: stop at once
            status = AVIP_ENAN;
            break;
          }
          if (it >= a.max_iter || (it > 0 && restarts >= kMaxRestarts)) {
            status = AVIP_ENOTCONV;
            break;
          }
          if (it > 0) ++restarts;
          fresh = true;
          check = false;
        }
        // ---- finest down phase on the residual, updated by the last step unless fresh:
        //      r' = r - alpha q, x += alpha p (own rows), r'.r'; xp0 = Q r', b1 = Rf r'
        {
          const double al = fresh ? 0.0 : alpha;
          const bool upd = !fresh;
          const double* __restrict__ rv = rc;
          const double* __restrict__ qv = a.q_ap;
          const T* __restrict__ trv = tc;
          const T* __restrict__ tqv = tq;
          const T alT = (T)al;
          // the gathered residual r - alpha q in the hierarchy's type
          auto res = [trv, tqv, alT, upd](int c) {
            return upd ? fma_t(-alT, __ldca(tqv + c), __ldca(trv + c)) : __ldca(trv + c);
          };
          double rr = 0.0;
          struct Pre {
            double r, q, x, p;
          };
          struct Hook {  // r' = r - alpha q into the other buffer (and its copy), x += alpha p, r'.r'
            const double *rv, *qv, *pv;
            double *xv, *rnv, *rr;
            T* tnv;
            double al;
            bool upd;
            __device__ Pre begin(int i) const {
              if (!upd) return Pre{0.0, 0.0, 0.0, 0.0};
              return Pre{__ldca(rv + i), __ldca(qv + i), xv[i], pv[i]};
            }
            __device__ void end(int i, const Pre& p) const {
              if (!upd) return;
              const double v = fma(-al, p.q, p.r);
              rnv[i] = v;
              if (kCopies) tnv[i] = (T)v;
              xv[i] = fma(al, p.p, p.x);
              *rr = fma(v, v, *rr);
            }
          } hook{rv, qv, a.p, a.x, rn, &rr, tn, al, upd};
          if (dl == 0) {
            for (int s = gwarp; s < nsl; s += nwarps) {
              const int i = s * kSlice + lane;
              if (i < N) hook.end(i, hook.begin(i));
            }
          } else {
            amg_down(C, ops, 0, [res](int c) { return (T)res(c); }, hook, gwarp, nwarps, lane);
          }
          if (upd) {
            double tot[1];
            if (!ops.template sum_epi<1>(rr, tot, check, [thresh](double t, double* o) {
                  o[0] = t;
                  return t <= thresh || !isfinite(t);
                }))
              return false;
            ++it;
            double* t = rc;
            rc = rn;
            rn = t;
            T* tt = tc;
            tc = tn;
            tn = tt;
            if (check) continue;  // confirm on the true residual
          } else if (!ops.barrier()) {
            return false;
          }
        }
        // ---- the levels below, then the finest up phase: z = U0 xp0 + Pf0 x1, r.z
        double rzb[2];  // r.z, beta
        bool positive;
        {
          DotAcc<double> acc;
          const double* __restrict__ rv = rc;
          struct Out {  // z_i = value (widened once here: w = A z gathers it in FP64), r_i z_i into r.z
            const double* rv;
            double* z;
            DotAcc<double>* acc;
            __device__ double begin(int i) const { return __ldca(rv + i); }
            __device__ void end(int i, T v, double ri) const {
              const double zi = (double)v;
              z[i] = zi;
              acc->add(ri, zi);
            }
          } out{rv, z, &acc};
          if (dl == 0) {
            const T* __restrict__ tv = tc;  // r in the hierarchy's type
            amg_dense(C, ops, [tv](int k) { return __ldca(tv + k); }, out, lane);
          } else {
            if (!amg_inner(C, ops, gwarp, nwarps, lane)) return false;
            amg_up(C, ops, 0, out, lane);
          }
          const double rz_old = rz;
          const bool first = fresh;
          if (!ops.template sum_epi<2>(acc.value(), rzb, positive, [rz_old, first](double t, double* o) {
                o[0] = t;
                o[1] = first ? 0.0 : t / rz_old;
                return t > 0.0 && isfinite(t);
              }))
            return false;
        }
        if (!positive) {  // the preconditioned residual lost positivity
          if (it == 0 || restarts >= kMaxRestarts) {
            status = AVIP_ENOTCONV;
            break;
          }
          check = true;
          continue;
        }
        const double beta = rzb[1];
        const bool first = fresh;
        rz = rzb[0];
        fresh = false;
        // ---- w = A z, q = w + beta q, p = z + beta p, p.q -> alpha
        double pq[1] = {0.0};
        {
          const double* __restrict__ zc = z;
          double* __restrict__ qv = a.q_ap;
          double* __restrict__ pv = a.p;
          T* __restrict__ tqw = tq;
          struct PreA {
            double z, q, p;
          };
          stream_rows<double, double>(
              ops.ring, mat, lane, [zc](int c) { return __ldca(zc + c); },
              [=](int i) { return PreA{__ldca(zc + i), qv[i], pv[i]}; },
              [&](int i, double w, const PreA& o) {
                const double qn = first ? w : fma(beta, o.q, w);  // (restart: old p, q unused)
                const double pn = first ? o.z : fma(beta, o.p, o.z);
                qv[i] = qn;
                if (kCopies) tqw[i] = (T)qn;
                pv[i] = pn;
                pq[0] = fma(pn, qn, pq[0]);
              });
        }
        double al[1];
        bool unused;
        const double rz_now = rz;
        if (!ops.template sum_epi<1>(pq[0], al, unused, [rz_now](double t, double* o) {
              o[0] = rz_now / t;
              return false;
            }))
          return false;
        alpha = al[0];
      }
    }
    // ---- phi = D^-1/2 x
    for (int s = gwarp; s < nsl; s += nwarps) {
      const int i = s * kSlice + lane;
      if (i < N) a.phi[i] = a.dsqinv[i] * a.x[i];
    }
    if (leader) {
      a.res->pcg_iters = it;
      advance_history(a);
      a.res->pcg_status = status;
      a.res->pcg_relres = bb[0] > 0.0 ? sqrt(rr_true / bb[0]) : 0.0;
      a.res->pcg_bnorm = sqrt(bb[0]);
      if (status != AVIP_OK && a.sc->status == AVIP_OK) a.sc->status = status;
    }
    return true;
  }
}


// Mixed-precision solve with the FP32 hierarchy (kind 10 and the batched mixed form): FP64
// outer residual and correction, FP32 inner CG preconditioned by the FP32 V-cycle.  As in
// amg_cg_solve the update r - alpha q, e += alpha p of an iteration is folded into the finest down
// phase of the next.
template <class Ops>
__device__ bool amg_mixed_solve(const PcgArgs& a, const AmgCtx<float>& C, Ops& ops, int gwarp, int nwarps, int lane,
                                bool leader) {
  const int N = a.A.N, nsl = a.A.nslices, dl = C.D.level;
  const double* nb = a.nbuf + (size_t)a.sc->parity * AVIP_MAX_SPECIES * a.Npad;
  float* rc = a.r32;   // current inner residual
  float* rn = a.rq32;  // the other buffer
  float* __restrict__ e32 = a.e32;
  float* __restrict__ p32 = a.p32;
  float* __restrict__ q32 = a.q32;
  float* __restrict__ z32 = a.z32;

  const double gain = C.gain;
  const int hist = history_length(a);
  double bb = 0.0;
  for (int s = gwarp; s < nsl; s += nwarps) {
    const int i = s * kSlice + lane;
    if (i >= N) continue;
    a.x[i] = a.dsq[i] * predict_phi(a, i, hist);
    double b;
    if (a.use_density_rhs) {
      double rho = 0.0;
      if (a.rhs_src)
        rho = a.rhs_src[i];
      else
        for (int k = 0; k < a.ns; ++k) rho = fma(a.q[k], nb[(size_t)k * a.Npad + i], rho);
      b = fma(a.rhs_scale[i], rho, gain * a.lift[i]);
      a.b[i] = b;
    } else {
      b = a.b[i];
    }
    if (a.rhs_scale[i] != 0.0) bb = fma(b, b, bb);  // free rows only: a Dirichlet row holds its value exactly
    else a.x[i] = b;  // a Dirichlet unit row takes its (possibly ramped) value exactly
  }
  double bs[2];  // b.b and the stopping threshold on r.r
  bool zero;
  {
    const double rtol = a.rtol;
    if (!ops.template sum_epi<2>(bb, bs, zero, [rtol](double t, double* o) {
          o[0] = t;
          o[1] = rtol * rtol * t;
          return t == 0.0;
        }))
      return false;
  }
  const double thresh = bs[1];
  int it = 0, outer = 0, status = AVIP_OK;
  double rr64 = 0.0;
  while (true) {
    // ---- FP64 residual of the FP64 iterate (x complete)
    double r2 = 0.0;
    for (int s = gwarp; s < nsl; s += nwarps) {
      const int i = s * kSlice + lane;
      if (i >= N) continue;
      const double r = a.b[i] - sell_row_dot(a.A, s, lane, i, a.x);
      a.r[i] = r;
      r2 = fma(r, r, r2);
    }
    double rs[3];  // r.r, its root and 1 / root
    bool small;
    if (!ops.template sum_epi<3>(r2, rs, small, [thresh](double t, double* o) {
          o[0] = t;
          o[1] = sqrt(t);
          o[2] = 1.0 / o[1];
          return t <= thresh;
        }))
      return false;
    rr64 = rs[0];
    if (!isfinite(rr64)) {
      status = AVIP_ENAN;
      break;
    }
    if (small || zero) break;
    if (it >= a.max_iter) {
      status = AVIP_ENOTCONV;
      break;
    }
    ++outer;
    const int it_outer = it;
    const double rnorm = rs[1], rscale = rs[2];
    // ---- FP32 right-hand side r / ||r||, e = 0
    double g0[2];  // its square norm, the inner stopping threshold
    bool go;
    {
      DotAcc<float> k;
      for (int s = gwarp; s < nsl; s += nwarps) {
        const int i = s * kSlice + lane;
        if (i >= N) continue;
        const float r = (float)(a.r[i] * rscale);
        rc[i] = r;
        e32[i] = 0.f;
        k.add(r, r);
      }
      const double in_rtol = a.inner_rtol;
      if (!ops.template sum_epi<2>(k.value(), g0, go, [in_rtol](double t, double* o) {
            o[0] = t;
            o[1] = in_rtol * in_rtol * t;
            return t > o[1];
          }))
        return false;
    }
    const double inner_thresh = g0[1];
    double rz = 0.0;
    float alpha = 0.f;
    bool fresh = true;
    while (go) {
      // ---- finest down phase on the residual, updated by the last step unless fresh
      {
        const float* __restrict__ rv = rc;
        const float al = alpha;
        const bool upd = !fresh;
        auto res = [rv, q32, al, upd](int c) {
          return upd ? fmaf(-al, __ldca(q32 + c), __ldca(rv + c)) : __ldca(rv + c);
        };
        DotAcc<float> krr;
        struct Pre {
          float r, q, e, p;
        };
        struct Hook {
          const float *rv, *qv, *pv;
          float *ev, *rnv;
          DotAcc<float>* krr;
          float al;
          bool upd;
          __device__ Pre begin(int i) const {
            if (!upd) return Pre{0.f, 0.f, 0.f, 0.f};
            return Pre{__ldca(rv + i), __ldca(qv + i), ev[i], pv[i]};
          }
          __device__ void end(int i, const Pre& p) const {
            if (!upd) return;
            const float v = fmaf(-al, p.q, p.r);
            rnv[i] = v;
            ev[i] = fmaf(al, p.p, p.e);
            krr->add(v, v);
          }
        } hook{rv, q32, p32, e32, rn, &krr, al, upd};
        if (dl == 0) {
          for (int s = gwarp; s < nsl; s += nwarps) {
            const int i = s * kSlice + lane;
            if (i < N) hook.end(i, hook.begin(i));
          }
        } else {
          amg_down(C, ops, 0, res, hook, gwarp, nwarps, lane);
        }
        if (upd) {
          double none[1];
          bool done;
          if (!ops.template sum_epi<1>(krr.value(), none, done, [inner_thresh](double t, double* o) {
                o[0] = t;
                return !(t > inner_thresh);
              }))
            return false;
          ++it;
          float* t = rc;
          rc = rn;
          rn = t;
          if (done || it >= a.max_iter) break;
        } else if (!ops.barrier()) {
          return false;
        }
      }
      // ---- the levels below, then the finest up phase: z = U0 xp0 + Pf0 x1, r.z
      double rzb[2];  // r.z, beta
      bool positive;
      {
        DotAcc<double> acc;
        struct Out {
          const float* rv;
          float* z;
          DotAcc<double>* acc;
          __device__ float begin(int i) const { return __ldca(rv + i); }
          __device__ void end(int i, float v, float ri) const {
            z[i] = v;
            acc->add((double)ri, (double)v);
          }
        } out{rc, z32, &acc};
        if (dl == 0) {
          const float* __restrict__ rv = rc;
          amg_dense(C, ops, [rv](int k) { return __ldca(rv + k); }, out, lane);
        } else {
          if (!amg_inner(C, ops, gwarp, nwarps, lane)) return false;
          amg_up(C, ops, 0, out, lane);
        }
        const double rz_old = rz;
        const bool first = fresh;
        if (!ops.template sum_epi<2>(acc.value(), rzb, positive, [rz_old, first](double t, double* o) {
              o[0] = t;
              o[1] = first ? 0.0 : t / rz_old;
              return t > 0.0 && isfinite(t);
            }))
          return false;
      }
      if (!positive) break;  // refine with what the inner solve has
      const float beta = (float)rzb[1];
      const bool first = fresh;
      rz = rzb[0];
      fresh = false;
      // ---- w = A z, q = w + beta q, p = z + beta p, p.q -> alpha
      DotAcc<float> kpq;
      struct PreA {
        float z, q, p;
      };
      stream_rows<float, float>(
          ops.ring, C.mat_phase(), lane, [z32](int c) { return __ldca(z32 + c); },
          [=](int i) { return PreA{__ldca(z32 + i), q32[i], p32[i]}; },
          [&](int i, float w, const PreA& o) {
            const float qn = first ? w : fmaf(beta, o.q, w);  // (restart: old p, q unused)
            const float pn = first ? o.z : fmaf(beta, o.p, o.z);
            q32[i] = qn;
            p32[i] = pn;
            kpq.add(pn, qn);
          });
      double al[1];
      bool unused;
      const double rz_now = rz;
      if (!ops.template sum_epi<1>(kpq.value(), al, unused, [rz_now](double t, double* o) {
            o[0] = rz_now / t;
            return false;
          }))
        return false;
      alpha = (float)al[0];
    }
    if (it == it_outer) {  // the inner solve could not start: no progress is possible
      status = AVIP_ENOTCONV;
      break;
    }
    // ---- FP64 correction x += ||r|| e
    for (int s = gwarp; s < nsl; s += nwarps) {
      const int i = s * kSlice + lane;
      if (i >= N) continue;
      a.x[i] = fma(rnorm, (double)e32[i], a.x[i]);
    }
    if (!ops.barrier()) return false;  // x complete before the next residual
  }
  for (int s = gwarp; s < nsl; s += nwarps) {
    const int i = s * kSlice + lane;
    if (i < N) a.phi[i] = a.dsqinv[i] * (zero ? a.b[i] : a.x[i]);  // free b == 0: x = b
  }
  if (leader) {
    a.res->pcg_iters = it;
    advance_history(a);
    a.res->pcg_outer = outer;
    a.res->pcg_status = status;
    a.res->pcg_relres = bs[0] > 0.0 ? sqrt(rr64 / bs[0]) : 0.0;
    a.res->pcg_bnorm = sqrt(bs[0]);
    if (status != AVIP_OK && a.sc->status == AVIP_OK) a.sc->status = status;
  }
  return true;
}


// Grid-wide synchronisation of a cooperative launch (counter barrier of grid_sync.cuh); MAXV: most
// values of one sum; kKeep: sums in the order the mixed-precision solves keep (block_group_sum).  sum_epi evaluates `epi(total, out)` on one thread per block: a division or
// comparison that every thread repeats costs a 1024-thread block 600 cycles per FP64 instruction
// (a division 5,000), one thread 64.  It returns a flag, and up to three derived scalars in out.
template <class R, int MAXV, bool kKeep = false>
struct GridOps {
  FlagSync& fs;
  R ring;
  __device__ bool barrier() { return grid_barrier<MAXV>(fs); }
  template <int NE, class Epi>
  __device__ bool sum_epi(double v, double (&out)[NE], bool& flag, Epi epi) {
    double s[1] = {v}, e[NE + 1];
    if (!grid_allsum<1, NE + 1, MAXV, kKeep>(s, e, fs, nullptr,
                                      [&epi](const double* t, double* o) { o[NE] = epi(t[0], o) ? 1.0 : 0.0; }))
      return false;
#pragma unroll
    for (int k = 0; k < NE; ++k) out[k] = e[k];
    flag = __double2hiint(e[NE]) != 0;
    return true;
  }
  __device__ bool sum(double (&v)[1]) {
    double e[1];
    return grid_allsum<1, 0, MAXV, kKeep>(v, e, fs, nullptr, NoEpilogue());
  }
};

// The two halves of a cluster barrier.  A solve passes one before its first write to another CTA's shared
// memory, which is there only once that CTA has started.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.aligned;" ::: "memory"); }

// Synchronisation of one thread-block cluster: hardware cluster barrier (release / acquire at
// cluster scope, so global-memory writes of the cluster are visible after it) and sums through
// distributed shared memory (at most 16 CTAs; deterministic: fixed order of threads and ranks).
// A CTA's partial is pushed into every CTA's table before the barrier, so that only local
// shared memory is read after it.
struct ClusterSums {
  double thr[1024];     // per-thread values
  double grp[4];
  double2 part[2][16];  // [parity][rank]: the CTA's sum and its SolveShared::bad
  double res[4];
  int flag;             // bit 0: the epilogue's, bit 1: a CTA gave up a wait
};
template <class R, bool kKeep = false>
struct ClusterOps {
  cooperative_groups::cluster_group cl;
  ClusterSums& sh;
  R ring;
  unsigned seq;
  const volatile int* bad;  // SolveShared::bad: travels with the sums, so that all CTAs leave at the same one
  __device__ bool barrier() {
    cluster_sync();
    return true;
  }
  // Cluster barrier with one releasing fence per CTA (after bar.sync, so it covers the writes of
  // all its threads) instead of one per thread: 2,250 -> 1,880 cycles at 16 x 512 threads with
  // stores in flight.
  __device__ void cluster_sync() {
    __syncthreads();
    if (threadIdx.x == 0) asm volatile("fence.acq_rel.cluster;" ::: "memory");
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
  template <int NE, class Epi>
  __device__ bool sum_epi(double v, double (&out)[NE], bool& flag, Epi epi) {
    static_assert(NE <= 4, "ClusterSums::res");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, C = (int)cl.num_blocks();
    const int par = (int)(seq++ & 1);
    double2* part = sh.part[par];
    double s[1] = {v}, bt[1];
    int lost;
    if constexpr (kKeep) {
      // the mixed-precision solves' order (see block_group_sum): a tree in every warp, then the
      // warps in turn
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s[0] += __shfl_xor_sync(0xffffffffu, s[0], o);
      if (lane == 0) sh.thr[warp] = s[0];
      __syncthreads();
      lost = *bad;
      if (warp == 0) {
        bt[0] = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) bt[0] += sh.thr[w];
      }
    } else {
      lost = block_group_sum<1>(s, bt, sh.thr, sh.grp, bad);
    }
    if (warp == 0 && lane < C) *cl.map_shared_rank(part + cl.block_rank(), lane) = make_double2(bt[0], lost ? 1.0 : 0.0);
    cluster_sync();
    if (warp == 0) {
      const double2 p = lane < C ? part[lane] : make_double2(0.0, 0.0);
      const bool any = __any_sync(0xffffffffu, __double2hiint(p.y) != 0);
      double t = p.x;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (lane == 0) sh.flag = (epi(t, sh.res) ? 1 : 0) | (any ? 2 : 0);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NE; ++k) out[k] = sh.res[k];
    const int f = sh.flag;
    flag = (f & 1) != 0;
    return f < 2;
  }
  // The first sum of amg_cg_solve, and its only one of this form.
  __device__ bool sum(double (&v)[1]) {
    cluster_wait();
    bool f;
    return sum_epi<1>(v[0], v, f, [](double t, double* o) {
      o[0] = t;
      return false;
    });
  }
};

}  // namespace avip
