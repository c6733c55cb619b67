// Drift-diffusion part of the explicit step, FP64, node-centric and atomic-free.
//
//   node_fields_kernel  E = -grad(phi), grad(n_s), nodal velocities V_s = sign(q_s) mu_s E,
//                       n_s mu_s, source rates, chemical time-step candidates
//   dt_cells_kernel     cell-based CFL / Fourier / dielectric candidates (section "Time step
//                       computation"); global minimum by an integer atomicMin on the bits of
//                       the positive doubles (exact and order independent)
//   flux_update_kernel  for each node, every incident edge flux (limited Lax-Wendroff +
//                       central diffusion) and the node-flux boundary closure, then source
//                       and explicit update into the other density buffer; per-block charge
//   finalize_kernel     charge sum in fixed order, time, parity flip, run statistics
//   *32 forms           the same in FP32 arithmetic for the mixed-precision path
//
// The residual of Eq. vertex_centered_flux is a sum over the edges of each dual cell.  Here
// every node gathers its own edges (each flux is evaluated at both ends), so no scatter and
// no atomics are needed and the result is deterministic.  Each edge flux is evaluated from the
// (lower index, higher index) ordered pair, so both ends compute bit-identical values and the
// scheme stays exactly conservative.
#include <cuda_runtime.h>

#include <cfloat>

#include "avip_internal.h"
#include "fp64_math.cuh"

namespace avip {

constexpr int kDDThreads = 256;
constexpr int kDDMinThreads = 128;  // smallest block of the batched stages (autotuned)

// Sign and magnitude tests on the bit patterns: an FP64 comparison costs as much as
// an FP64 multiply-add (19 cycles per warp and SM), integer ones next to nothing.
__device__ __forceinline__ long long abs_bits(double x) { return __double_as_longlong(x) & 0x7fffffffffffffffLL; }
__device__ __forceinline__ bool negative(double x) { return __double2hiint(x) < 0; }
__device__ __forceinline__ double flip_sign(double x, bool flip) {
  return __hiloint2double(__double2hiint(x) ^ (flip ? (int)0x80000000 : 0), __double2loint(x));
}

// Local-field mobility and the Townsend exponential with the library's FP64 exp / log
// (fp64_math.cuh: a few ulp, a fraction of the FP64 instructions of the general routines).
// mu0 (max(|E|, E_floor) / E_ref)^p = mu0 exp(p (log max(|E|, E_floor) - log E_ref)), log E_ref
// from the host: no FP64 division.
__device__ __forceinline__ double mobility(const SpeciesParams& sp, double Emag) {
  if (sp.mob_model == AVIP_MOB_POWER)
    return sp.mob[0] * exp_fp64(sp.mob[2] * (log_fp64(abs_bits(Emag) < abs_bits(sp.mob[3]) ? sp.mob[3] : Emag) -
                                             sp.mob_log_ref));
  return sp.mob[0];
}

__device__ __forceinline__ double limiter(double r, double beta, int kind) {
  if (kind == AVIP_LIM_VANLEER) {
    if (abs_bits(r) == 0x7ff0000000000000LL) return negative(r) ? 0.0 : 2.0;  // (an overflowed ratio)
    return (r + fabs(r)) / (1.0 + fabs(r));
  }
  return fmax(0.0, fmax(fmin(beta * r, 1.0), fmin(r, beta)));
}

// num / delta, delta != 0: through the Newton reciprocal, or the division where delta is subnormal.  An
// explicit front that runs into a zero background decays through the subnormals, and 1 / delta
// overflows below 2^-1024.
__device__ __forceinline__ double slope_ratio(double num, double delta) {
  if (abs_bits(delta) < 0x0010000000000000LL) return num / delta;
  return num * recip_nr(delta);
}

// Smallest positive v of the block into *dst (the bits of positive doubles order like integers):
// two integer warp reductions, no FP64 comparison (each costs the SM 19 cycles per warp).
__device__ __forceinline__ void block_min_to_global(double v, unsigned long long* dst) {
  __shared__ unsigned long long sm[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  constexpr unsigned long long kInf = 0x7ff0000000000000ULL;
  const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
  const unsigned long long key = bits == 0 || bits > kInf ? kInf : bits;  // zero, negative, NaN: no candidate
  auto warp_min = [](unsigned long long k) {
    const unsigned hi = __reduce_min_sync(0xffffffffu, (unsigned)(k >> 32));
    const unsigned lo = __reduce_min_sync(0xffffffffu, (unsigned)(k >> 32) == hi ? (unsigned)k : 0xffffffffu);
    return (unsigned long long)hi << 32 | lo;
  };
  const unsigned long long w = warp_min(key);
  if (lane == 0) sm[warp] = w;
  __syncthreads();
  if (warp == 0) {
    const unsigned long long t = warp_min(lane < nw ? sm[lane] : kInf);
    if (lane == 0 && t < kInf) atomicMin(dst, t);
  }
}

// ------------------------------------------------------------------------ nodal fields
__device__ __forceinline__ void node_fields_body(const DDArgs& a, int with_dt, int bid) {
  const int i = bid * blockDim.x + threadIdx.x;
  const int N = a.A.N;
  const int ns = a.ph.ns;
  double chem = INFINITY;
  if (i < N) {
    const int slice = i / kSlice, lane = i % kSlice;
    const double* n = a.nbuf + (size_t)a.sc->parity * AVIP_MAX_SPECIES * a.Npad;
    const int base = __ldg(a.A.sl_ptr + slice) + lane;
    const int rl = __ldg(a.A.rlen + i);
    double gpx = 0.0, gpy = 0.0;
    double gnx[AVIP_MAX_SPECIES], gny[AVIP_MAX_SPECIES];
#pragma unroll
    for (int s = 0; s < AVIP_MAX_SPECIES; ++s) gnx[s] = gny[s] = 0.0;
    // neighbours in groups of kG: the column and weight loads of a group are issued together,
    // then its potential and density gathers, then the sums (in slot order, as one at a time)
    constexpr int kG = 4;
    for (int k0 = 0; k0 < rl; k0 += kG) {
      int c[kG];
      double wx[kG], wy[kG];
#pragma unroll
      for (int u = 0; u < kG; ++u) {
        const int e = base + (k0 + u) * kSlice;
        const bool in = k0 + u < rl;
        c[u] = in ? __ldg(a.A.col + e) : i;
        wx[u] = in ? __ldg(a.A.gx + e) : 0.0;
        wy[u] = in ? __ldg(a.A.gy + e) : 0.0;
      }
      double pj[kG];
#pragma unroll
      for (int u = 0; u < kG; ++u) pj[u] = a.phi[c[u]];
#pragma unroll
      for (int u = 0; u < kG; ++u) {
        if (k0 + u < rl) {
          gpx = fma(wx[u], pj[u], gpx);
          gpy = fma(wy[u], pj[u], gpy);
        }
      }
#pragma unroll
      for (int s = 0; s < AVIP_MAX_SPECIES; ++s) {
        if (s < ns && !a.ph.sp[s].immobile) {
          double uj[kG];
#pragma unroll
          for (int u = 0; u < kG; ++u) uj[u] = n[(size_t)s * a.Npad + c[u]];
#pragma unroll
          for (int u = 0; u < kG; ++u) {
            if (k0 + u < rl) {
              gnx[s] = fma(wx[u], uj[u], gnx[s]);
              gny[s] = fma(wy[u], uj[u], gny[s]);
            }
          }
        }
      }
    }
    const double Ex = -gpx, Ey = -gpy;
    // |E| and 1/|E| from one reciprocal square root (the Townsend and attachment exponents take
    // -B/|E| as a product)
    const double E2 = Ex * Ex + Ey * Ey;
    const double invE = abs_bits(E2) != 0 ? rsqrt(E2) : 0.0;
    const double Emag = E2 * invE;
    a.Ex[i] = Ex;
    a.Ey[i] = Ey;
    double mu[AVIP_MAX_SPECIES];
#pragma unroll
    for (int s = 0; s < AVIP_MAX_SPECIES; ++s) {
      if (s < ns) {
        const SpeciesParams& sp = a.ph.sp[s];
        mu[s] = mobility(sp, Emag);
        const double sg = sp.q > 0 ? 1.0 : -1.0;
        const double vx = sg * mu[s] * Ex, vy = sg * mu[s] * Ey;
        double2* d = reinterpret_cast<double2*>(a.ndat + ((size_t)s * a.Npad + i) * 4);
        d[0] = make_double2(gnx[s], gny[s]);
        d[1] = make_double2(vx, vy);
        const double nmu = n[(size_t)s * a.Npad + i] * mu[s];
        a.nm[(size_t)s * a.Npad + i] = nmu;
        a.vf[(size_t)s * a.Npad + i] = make_float4((float)vx, (float)vy, (float)nmu, 0.f);
      }
    }
    double src[AVIP_MAX_SPECIES];
#pragma unroll
    for (int s = 0; s < AVIP_MAX_SPECIES; ++s) src[s] = 0.0;
    if (a.ph.src_model != AVIP_SRC_NONE) {
      const int ie = a.ph.src_idx[0], ip = a.ph.src_idx[1], ineg = a.ph.src_idx[2];
      const double ne = n[(size_t)ie * a.Npad + i];
      const double alpha = abs_bits(Emag) != 0 ? a.ph.src_params[0] * exp_fp64(-a.ph.src_params[1] * invE) : 0.0;
      double mue = 0.0;
#pragma unroll
      for (int s = 0; s < AVIP_MAX_SPECIES; ++s)
        if (s == ie) mue = mu[s];
      const double ion = alpha * mue * Emag * ne;
      if (a.ph.photo_terms > 0) a.photo_I[i] = ion;
#pragma unroll
      for (int s = 0; s < AVIP_MAX_SPECIES; ++s) {
        if (s == ie) src[s] += ion;
        if (s == ip) src[s] += ion;
      }
      if (a.ph.src_model == AVIP_SRC_TOWNSEND_ATTACH) {
        const double att = a.ph.src_params[2] * ne;
#pragma unroll
        for (int s = 0; s < AVIP_MAX_SPECIES; ++s) {
          if (s == ie) src[s] -= att;
          if (s == ineg) src[s] += att;
        }
      } else if (a.ph.src_model == AVIP_SRC_MORROW_LOWKE) {
        // attachment eta(|E|) w n_e, recombination beta_r n_e n_p and beta_r n_n n_p
        double npos = 0.0, nneg = 0.0;
#pragma unroll
        for (int s = 0; s < AVIP_MAX_SPECIES; ++s) {
          if (s == ip) npos = n[(size_t)s * a.Npad + i];
          if (s == ineg) nneg = n[(size_t)s * a.Npad + i];
        }
        const double eta = abs_bits(Emag) != 0 ? a.ph.src_params[2] * exp_fp64(-a.ph.src_params[3] * invE) : 0.0;
        const double att = eta * mue * Emag * ne;
        const double rep = a.ph.src_params[4] * ne * npos;
        const double rnp = a.ph.src_params[4] * nneg * npos;
#pragma unroll
        for (int s = 0; s < AVIP_MAX_SPECIES; ++s) {
          if (s == ie) src[s] = src[s] - att - rep;
          if (s == ip) src[s] = src[s] - rep - rnp;
          if (s == ineg) src[s] = src[s] + att - rnp;
        }
      }
      double se = 0.0;
#pragma unroll
      for (int s = 0; s < AVIP_MAX_SPECIES; ++s)
        if (s == ie) se = src[s];
      if (abs_bits(se) != 0) chem = a.ph.a_chem * fabs(ne) * recip_nr(fabs(se));
    }
#pragma unroll
    for (int s = 0; s < AVIP_MAX_SPECIES; ++s)
      if (s < ns) a.src[(size_t)s * a.Npad + i] = src[s];
  }
  if (with_dt) block_min_to_global(chem, &a.sc->dt_bits);
}

// The kernels of a single-instance step are launched with programmatic stream serialisation: each is
// put on the SMs while its predecessor drains and waits here, before it reads anything, until the
// predecessor has completed and its writes are visible.  Hides the launch of four of the step's
// kernels, which dominate it on small meshes.
__device__ __forceinline__ void after_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__global__ void __launch_bounds__(kDDThreads, 3) node_fields_kernel(DDArgs a, int with_dt) {
  after_predecessor();
  node_fields_body(a, with_dt, blockIdx.x);
}

// ------------------------------------------------------------------------ time step
// Convective and dielectric limits over cells (section "Time step computation"), with the cell
// velocity and conductivity the means of the n_v nodal values.  Each thread carries the largest
// |V_cell| / dx (the sum of the nodal velocities times the per-cell weight 1/(n_v dx)) and the
// largest conductivity over its cells and species, and divides once at the end:
// min_c cfl dx / |V| = cfl / max_c |V| / dx, likewise for the dielectric limit.  The Fourier
// limit, fourier dx^2 / D over cells and species, depends on the mesh only (ph.dt_fourier).
//
// The two maxima are screened in FP32: every cell's |V_cell| / dx and conductivity get a lower and an
// upper bound from FP32 copies of the nodal values (a.vf, written by the nodal kernel: vx, vy,
// n mu) and a bound of the FP32 rounding, and only the cells whose upper bound reaches the
// block's largest lower bound, in blocks that can still lower the global minimum, are evaluated
// in FP64.  The cell that sets the time step always is, so the result is the FP64 one bit for
// bit.  On GB300 the FP64 pipe bounded this kernel (16 operations per cell and species; 997,002
// triangles, 2 species: 93 us).
constexpr int kDtCells = 4;  // cells per thread
__device__ __forceinline__ void dt_cell_fp64(const DDArgs& a, int c, double& v2max, double& smax) {
  const int ns = a.ph.ns;
  const int n0 = a.cell[c], n1 = a.cell[a.T + c], n2 = a.cell[2 * a.T + c];
  const int n3 = a.nvmax == 4 ? a.cell[3 * a.T + c] : -1;  // -1: triangle
  const bool quad = n3 >= 0;
  const double w = a.cw[c], w2 = w * w;
  const double inv_nv = quad ? 0.25 : (1.0 / 3.0);
  double sigma = 0.0;
  for (int s = 0; s < ns; ++s) {
    double vx, vy;
    if (a.ph.dd_fp32) {  // FP32 velocities, FP64 candidate and reduction
      const float* d = a.ndat32 + (size_t)s * a.Npad * 4;
      vx = (double)d[4 * n0 + 2] + (double)d[4 * n1 + 2] + (double)d[4 * n2 + 2];
      vy = (double)d[4 * n0 + 3] + (double)d[4 * n1 + 3] + (double)d[4 * n2 + 3];
      if (quad) {
        vx += (double)d[4 * n3 + 2];
        vy += (double)d[4 * n3 + 3];
      }
    } else {
      const double* d = a.ndat + (size_t)s * a.Npad * 4;
      vx = d[4 * n0 + 2] + d[4 * n1 + 2] + d[4 * n2 + 2];
      vy = d[4 * n0 + 3] + d[4 * n1 + 3] + d[4 * n2 + 3];
      if (quad) {
        vx += d[4 * n3 + 2];
        vy += d[4 * n3 + 3];
      }
    }
    v2max = fmax(v2max, (vx * vx + vy * vy) * w2);
    const double* nm = a.nm + (size_t)s * a.Npad;
    double cell = nm[n0] + nm[n1] + nm[n2];
    if (quad) cell += nm[n3];
    sigma += fabs(a.ph.sp[s].q * kECharge * cell);
  }
  smax = fmax(smax, sigma * inv_nv);
}

__device__ __forceinline__ void dt_cells_body(const DDArgs& a, int bid, int nblocks) {
  __shared__ unsigned long long s_max[2];  // bits of the block's FP64 maxima
  __shared__ unsigned s_lo[2];             // bits of the block's largest FP32 lower bounds
  __shared__ float s_cur;
  const int ns = a.ph.ns, stride = nblocks * blockDim.x;
  constexpr float kEps = 1e-6f;  // FP32 rounding of the sums below, relative to the sum of magnitudes
  // below this the squares (and sums) come near FP32's subnormals, where kEps does not bound their
  // rounding: such a cell counts as this large above and as nothing below
  constexpr float kTiny = 1e-30f;
  if (threadIdx.x < 2) {
    s_max[threadIdx.x] = 0;
    s_lo[threadIdx.x] = 0;
  }
  // the running minimum over the blocks already done, rounded up (it only falls)
  double cur = 0.0;
  if (threadIdx.x == 0) cur = __longlong_as_double(*(volatile long long*)&a.sc->dt_bits);
  __syncthreads();
  for (int base = bid * blockDim.x + threadIdx.x; base - (int)threadIdx.x < a.T; base += kDtCells * stride) {
    float vhi[kDtCells], shi[kDtCells];  // upper bounds of (|V_cell| / dx) and of the conductivity
    float vlo = 0.f, slo = 0.f;
#pragma unroll
    for (int k = 0; k < kDtCells; ++k) {
      const int c = base + k * stride;
      vhi[k] = shi[k] = -1.f;
      if (c >= a.T || c < base) continue;
      const int n0 = __ldg(a.cell + c), n1 = __ldg(a.cell + a.T + c), n2 = __ldg(a.cell + 2 * a.T + c);
      const int n3 = a.nvmax == 4 ? __ldg(a.cell + 3 * a.T + c) : -1;
      const float w = __ldg(a.cw32 + c);
      float v = 0.f, vl = 0.f, sig = 0.f, sige = 0.f;
      for (int s = 0; s < ns; ++s) {
        const float4* f = a.vf + (size_t)s * a.Npad;
        const float4 p0 = f[n0], p1 = f[n1], p2 = f[n2];
        float4 p3 = make_float4(0.f, 0.f, 0.f, 0.f);
        if (n3 >= 0) p3 = f[n3];
        const float vx = fabsf((p0.x + p1.x) + (p2.x + p3.x)), vy = fabsf((p0.y + p1.y) + (p2.y + p3.y));
        const float ex = kEps * ((fabsf(p0.x) + fabsf(p1.x)) + (fabsf(p2.x) + fabsf(p3.x)));
        const float ey = kEps * ((fabsf(p0.y) + fabsf(p1.y)) + (fabsf(p2.y) + fabsf(p3.y)));
        const float hx = (vx + ex) * w, hy = (vy + ey) * w;
        const float lx = fmaxf(vx - ex, 0.f) * w, ly = fmaxf(vy - ey, 0.f) * w;
        // !(x <= v): a NaN becomes an upper bound that no test excludes
        const float h2 = hx * hx + hy * hy;
        if (!(h2 <= v)) v = h2;
        vl = fmaxf(vl, lx * lx + ly * ly);
        sig += fabsf((p0.z + p1.z) + (p2.z + p3.z));
        sige += kEps * ((fabsf(p0.z) + fabsf(p1.z)) + (fabsf(p2.z) + fabsf(p3.z)));
      }
      const float inv_nv = n3 >= 0 ? 0.25f : 1.f / 3.f;
      if (v < kTiny) v = kTiny;
      sige += kTiny;
      vhi[k] = v * (1.f + 4.f * kEps);
      if (vl >= kTiny) vlo = fmaxf(vlo, vl * (1.f - 4.f * kEps));
      shi[k] = (sig + sige) * inv_nv * (1.f + 4.f * kEps);
      slo = fmaxf(slo, fmaxf(sig - sige, 0.f) * inv_nv * (1.f - 4.f * kEps));
    }
    // the block's largest lower bounds (bits of nonnegative floats order like integers)
    const unsigned bv = __reduce_max_sync(0xffffffffu, __float_as_uint(vlo));
    const unsigned bs = __reduce_max_sync(0xffffffffu, __float_as_uint(slo));
    if ((threadIdx.x & 31) == 0) {
      if (bv) atomicMax(&s_lo[0], bv);
      if (bs) atomicMax(&s_lo[1], bs);
    }
    if (threadIdx.x == 0) s_cur = __double2float_ru(cur);
    __syncthreads();
    const float now = s_cur, cfl = (float)a.ph.cfl, diel = (float)a.ph.a_diel * (float)(kEps0 / kECharge);
    const float vthr = __uint_as_float(s_lo[0]), sthr = __uint_as_float(s_lo[1]);
#pragma unroll
    for (int k = 0; k < kDtCells; ++k) {
      const int c = base + k * stride;
      if (c >= a.T || c < base) continue;
      const bool ev = !(vhi[k] < vthr) && !(cfl * rsqrtf(vhi[k]) * (1.f - 1e-5f) > now);
      const bool es = !(shi[k] < sthr) && !(diel / shi[k] * (1.f - 1e-5f) > now);
      if (ev || es) {
        double v2 = 0.0, sm = 0.0;
        dt_cell_fp64(a, c, v2, sm);
        if (v2 > 0.0) atomicMax(&s_max[0], (unsigned long long)__double_as_longlong(v2));
        if (sm > 0.0) atomicMax(&s_max[1], (unsigned long long)__double_as_longlong(sm));
      }
    }
  }
  __syncthreads();
  // one thread per limit, in different warps (a square root or a division takes 650 cycles)
  if ((threadIdx.x & 31) == 0 && threadIdx.x < 96) {
    const int k = threadIdx.x >> 5;
    double cand = a.ph.dt_fourier;
    if (k < 2) {
      const double m = __longlong_as_double((long long)s_max[k]);
      cand = !(m > 0.0) ? INFINITY : k == 0 ? a.ph.cfl / sqrt(m) : a.ph.a_diel * kEps0 / m;
    }
    if (cand > 0.0 && cand < INFINITY) atomicMin(&a.sc->dt_bits, (unsigned long long)__double_as_longlong(cand));
  }
}

__global__ void __launch_bounds__(kDDThreads) dt_cells_kernel(DDArgs a) {
  after_predecessor();
  dt_cells_body(a, blockIdx.x, gridDim.x);
}

// ------------------------------------------------------------------------ fluxes + update
struct EdgeEnd {
  double u, gx, gy, vx, vy;
};

// Bernoulli function B(x) = x / (e^x - 1) for x >= 0 (B(0) = 1; 0 where it is below 1e-300).
// B(-x) = x + B(x), so one expm1 gives both values without cancellation.
__device__ __forceinline__ double bernoulli_pos(double x) {
  if (__double2hiint(x) < 0x3c300000) return 1.0;  // below 2^-60: 1 - x/2 rounds to 1 (and 1 / x may overflow)
  return x > 700.0 ? 0.0 : quotient_nr(x, expm1(x));
}

// Geometry of one edge for the Scharfetter-Gummel split (species independent), canonical
// orientation lo -> hi: edge vector d = h e, S.e / h = S.d / d.d and S_perp = S - (S.e) e.
struct SgGeo {
  double dx, dy, sh, spx, spy;
};
__device__ __forceinline__ SgGeo sg_geometry(double dx, double dy, double Sx, double Sy) {
  SgGeo g;
  g.dx = dx;
  g.dy = dy;
  g.sh = quotient_nr(fma(Sx, dx, Sy * dy), fma(dx, dx, dy * dy));
  g.spx = fma(-g.sh, dx, Sx);
  g.spy = fma(-g.sh, dy, Sy);
  return g;
}

// Scharfetter-Gummel flux (section "Scharfetter Gummel scheme"): S is split along the edge
// direction e into S_par = (S.e) e and S_perp; the tangential part is the exponentially fitted
// V.S_par (u_hi - e^a u_lo)/(1 - e^a), a = h V.e / D = V.d / D, evaluated as
// (D (S.e)/h)(B(-a) u_lo - B(a) u_hi) (no overflow for large |a|, no 0/0 at a = 0; D = 0 is
// the upwind limit); the normal part is centred: V.S_perp (u_lo + u_hi)/2 - D g.S_perp.  V and g
// come doubled (the sums of the two ends).  Written on d instead of e and h it needs no square
// root, and 1 / D comes from the host: fluxes and update of 313,000 edges, 2 species, 127 -> 94 us.
__device__ __forceinline__ double sg_flux(double ulo, double uhi, const SgGeo& G, double sVx, double sVy, double sgx,
                                          double sgy, const SpeciesParams& sp) {
  const double Vd = 0.5 * fma(sVx, G.dx, sVy * G.dy);  // V.d
  double fpar;
  if (sp.invD > 0.0) {  // (else the upwind limit: also for D below 2^-1024, whose part of the flux is nothing)
    const double a = Vd * sp.invD;
    const double aa = fabs(a);
    const double Bp = bernoulli_pos(aa), Bm = aa + Bp;  // B(|a|), B(-|a|)
    const bool neg = negative(a);
    fpar = (sp.D * G.sh) * fma(neg ? Bp : Bm, ulo, -((neg ? Bm : Bp) * uhi));
  } else {
    fpar = G.sh * Vd * (negative(Vd) ? uhi : ulo);
  }
  return fma(0.25 * fma(sVx, G.spx, sVy * G.spy), ulo + uhi, fma(-0.5 * sp.D, fma(sgx, G.spx, sgy * G.spy), fpar));
}

// Sum of the block's values into *dst in a fixed order: the warps' values through shared memory to
// one warp, which adds a column each and finishes with a shuffle tree (nw + 4 warp-wide FP64 adds
// instead of the 5 nw + 5 of a tree in every warp).
__device__ __forceinline__ void block_charge(double q, double* dst) {
  __shared__ double thr[kDDThreads];
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  thr[threadIdx.x] = q;
  __syncthreads();
  if (threadIdx.x < 32) {
    double t = thr[lane];
    for (int w = 1; w < nw; ++w) t += thr[w * 32 + lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) *dst = t;
  }
}

// Flux from `lo` to `hi` through the dual face with normal 2 (Hx, Hy) oriented lo -> hi:
// limited Lax-Wendroff convective part with a virtual upwind node plus central diffusion, or
// (sg != nullptr) the Scharfetter-Gummel flux.  (dx, dy) = x_hi - x_lo, dt4 = dt / 4.
//
// The edge means V_ij = (V_i + V_j)/2 and grad_ij = (grad_i + grad_j)/2 are kept as sums and the
// halves folded into the half normals and into psi / 2: scaling by a power of two is exact, so
// this adds no rounding.  23 FP64 operations per edge and species (33 with the halves, the sign
// and range tests and the coordinate differences in FP64): the FP64 issue rate bounds the kernel
// on GB300.
__device__ __forceinline__ double edge_flux(const EdgeEnd& lo, const EdgeEnd& hi, double dx, double dy, double Hx,
                                            double Hy, const SpeciesParams& sp, double dt4, double beta, int lim,
                                            const SgGeo* sg) {
  const double sVx = lo.vx + hi.vx, sVy = lo.vy + hi.vy;  // 2 V_ij
  const double sgx = lo.gx + hi.gx, sgy = lo.gy + hi.gy;  // 2 grad_ij
  if (sg) return sg_flux(lo.u, hi.u, *sg, sVx, sVy, sgx, sgy, sp);
  const double av = fma(sVx, Hx, sVy * Hy);               // V_ij . S
  const bool up_hi = negative(av);                        // (-0: no flux either way)
  const double uU = up_hi ? hi.u : lo.u;
  const double gU = fma(up_hi ? hi.gx : lo.gx, dx, (up_hi ? hi.gy : lo.gy) * dy);  // grad_U . (x_hi - x_lo)
  const double d = hi.u - lo.u;
  const double delta = flip_sign(d, up_hi);               // u_W - u_U
  const double num = fma(flip_sign(2.0, up_hi), gU, -delta);  // 2 grad_U . (x_W - x_U) - delta = r delta
  double hpsi = 0.0;                                      // psi / 2
  const long long ad = abs_bits(delta), an = abs_bits(num);
  if (lim == AVIP_LIM_SWEBY && beta == 1.0) {  // min-mod: psi = clamp(r, 0, 1)
    const bool same = ((__double2hiint(delta) ^ __double2hiint(num)) >= 0);
    if (ad != 0 && same) hpsi = an >= ad ? 0.5 : 0.5 * slope_ratio(num, delta);
  } else if (ad != 0) {
    hpsi = 0.5 * limiter(slope_ratio(num, delta), beta, lim);
  }
  const double lw = fma(-dt4, fma(sgx, sVx, sgy * sVy), delta);  // delta - dt grad_ij.V_ij
  const double us = fma(lw, hpsi, uU);
  return fma(us, av, -sp.D * fma(sgx, Hx, sgy * Hy));               // minus D grad_ij . S
}

// kGather: the edge fluxes were evaluated once per edge (edge_flux_kernel) and are gathered;
// otherwise every row evaluates its own edges (batches).  Specialised so that the single-instance
// kernel carries none of the per-row evaluation's registers.
template <bool kGather>
__device__ __forceinline__ void flux_update_body_t(const DDArgs& a, int bid) {
  const int i = bid * blockDim.x + threadIdx.x;
  const int N = a.A.N;
  const int ns = a.ph.ns;
  const double dt = a.ph.dt_fixed > 0.0 ? a.ph.dt_fixed : __longlong_as_double((long long)a.sc->dt_bits);
  const double dt4 = 0.25 * dt;
  double qsum = 0.0;
  if (i < N) {
    const int par = a.sc->parity;
    const double* n = a.nbuf + (size_t)par * AVIP_MAX_SPECIES * a.Npad;
    double* nn = a.nbuf + (size_t)(par ^ 1) * AVIP_MAX_SPECIES * a.Npad;
    const int slice = i / kSlice, lane = i % kSlice;
    const int base = __ldg(a.A.sl_ptr + slice) + lane;
    const int rl = __ldg(a.flen + i);  // edge slots only
    const double xi = kGather ? 0.0 : a.x[i], yi = kGather ? 0.0 : a.y[i];
    double R[AVIP_MAX_SPECIES];
    EdgeEnd me[AVIP_MAX_SPECIES];
#pragma unroll
    for (int s = 0; s < AVIP_MAX_SPECIES; ++s) {
      R[s] = 0.0;
      if (s < ns) {
        double2 g = make_double2(0.0, 0.0), v = g;
        if (!kGather) {  // (the gathering form reads the record of a boundary row only)
          const double2* d = reinterpret_cast<const double2*>(a.ndat + ((size_t)s * a.Npad + i) * 4);
          g = d[0];
          v = d[1];
        }
        me[s] = EdgeEnd{n[(size_t)s * a.Npad + i], g.x, g.y, v.x, v.y};
      }
    }
    if (kGather) {
      // fluxes already evaluated once per edge (lo -> hi), gathered in the same slot order: the
      // edge ids of kG slots are loaded together, then their fluxes, then summed in slot order
      constexpr int kG = 4;
      for (int k0 = 1; k0 < rl; k0 += kG) {
        int32_t v[kG];
#pragma unroll
        for (int u = 0; u < kG; ++u) v[u] = k0 + u < rl ? __ldg(a.slot_eid + base + (k0 + u) * kSlice) : 0;
#pragma unroll
        for (int s = 0; s < AVIP_MAX_SPECIES; ++s) {
          if (s < ns && !a.ph.sp[s].immobile) {
            double F[kG];
#pragma unroll
            for (int u = 0; u < kG; ++u) F[u] = k0 + u < rl ? a.eflux[(size_t)s * a.E + (v[u] & 0x7fffffff)] : 0.0;
#pragma unroll
            for (int u = 0; u < kG; ++u)
              if (k0 + u < rl) R[s] += flip_sign(F[u], v[u] >= 0);  // (the row is the lo end: flux out)
          }
        }
      }
    }
    for (int k = 1; k < (kGather ? 0 : rl); ++k) {
      const int e = base + k * kSlice;
      const int j = __ldg(a.A.col + e);
      const double Sx = __ldg(a.A.sx + e), Sy = __ldg(a.A.sy + e);
      const bool lo_is_me = i < j;
      // canonical lo -> hi: the stored normal and the difference below are oriented i -> j
      const double dx = flip_sign(a.x[j] - xi, !lo_is_me), dy = flip_sign(a.y[j] - yi, !lo_is_me);
      const double Hx = flip_sign(0.5 * Sx, !lo_is_me), Hy = flip_sign(0.5 * Sy, !lo_is_me);
      SgGeo geo;
      const bool use_sg = a.ph.scheme == AVIP_FLUX_SG;
      if (use_sg) geo = sg_geometry(dx, dy, 2.0 * Hx, 2.0 * Hy);
#pragma unroll
      for (int s = 0; s < AVIP_MAX_SPECIES; ++s) {
        if (s < ns && !a.ph.sp[s].immobile) {
          const double2* d = reinterpret_cast<const double2*>(a.ndat + ((size_t)s * a.Npad + j) * 4);
          const double2 g = d[0], v = d[1];
          const EdgeEnd other{n[(size_t)s * a.Npad + j], g.x, g.y, v.x, v.y};
          const EdgeEnd& lo = lo_is_me ? me[s] : other;
          const EdgeEnd& hi = lo_is_me ? other : me[s];
          const double F = edge_flux(lo, hi, dx, dy, Hx, Hy, a.ph.sp[s], dt4, a.ph.beta, a.ph.limiter,
                                     use_sg ? &geo : nullptr);
          R[s] += flip_sign(F, lo_is_me);
        }
      }
    }
    // boundary closure through the boundary nodal normal kept in the diagonal slot
    // (an interior row's S_i^b is exactly zero and its closure term with it)
    const double Sbx = __ldg(a.A.sx + base), Sby = __ldg(a.A.sy + base);
    const bool rim = (abs_bits(Sbx) | abs_bits(Sby)) != 0;
    const double Vi = a.vol[i], iVi = a.ivol[i];
    bool bad = false;
#pragma unroll
    for (int s = 0; s < AVIP_MAX_SPECIES; ++s) {
      if (s < ns) {
        const SpeciesParams& sp = a.ph.sp[s];
        double rs = R[s];
        if (rim) {
          const double2* d = reinterpret_cast<const double2*>(a.ndat + ((size_t)s * a.Npad + i) * 4);
          const double2 g = d[0], v = d[1];
          double Fx = me[s].u * v.x, Fy = me[s].u * v.y;
          if (sp.bnd_mode == AVIP_BND_OUTFLOW) {
            Fx -= sp.D * g.x;
            Fy -= sp.D * g.y;
          }
          rs -= Fx * Sbx + Fy * Sby;
        }
        const double un = me[s].u + dt * fma(rs, iVi, a.src[(size_t)s * a.Npad + i]);
        nn[(size_t)s * a.Npad + i] = un;
        bad |= (__double2hiint(un) & 0x7ff00000) == 0x7ff00000;
        qsum = fma(flip_sign(Vi, negative(sp.q)), un, qsum);  // charge numbers are -1 or +1
      }
    }
    if (bad) atomicCAS(&a.sc->status, AVIP_OK, AVIP_ENAN);
  }
  block_charge(qsum, a.partials + bid);
  if (bid == 0 && threadIdx.x == 0) a.sc->dt = dt;
}

template <bool kGather>
__global__ void __launch_bounds__(kDDThreads, kGather ? 3 : 2) flux_update_kernel(DDArgs a) {
  after_predecessor();
  flux_update_body_t<kGather>(a, blockIdx.x);
}

// One thread per edge (lo, hi): the flux of every species from lo to hi through the edge's dual
// face, the same function of the same operands as in flux_update_body's per-row evaluation, so
// both ends receive identical values.
__global__ void __launch_bounds__(kDDThreads) edge_flux_kernel(DDArgs a) {
  after_predecessor();
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= a.E) return;
  const int ns = a.ph.ns;
  const double dt4 = 0.25 * (a.ph.dt_fixed > 0.0 ? a.ph.dt_fixed : __longlong_as_double((long long)a.sc->dt_bits));
  const double* n = a.nbuf + (size_t)a.sc->parity * AVIP_MAX_SPECIES * a.Npad;
  const int lo = __ldg(a.e_lo + e), hi = __ldg(a.e_hi + e);
  const double Hx = __ldg(a.e_hx + e), Hy = __ldg(a.e_hy + e);  // half normal
  const double dx = __ldg(a.e_dx + e), dy = __ldg(a.e_dy + e);
  const bool use_sg = a.ph.scheme == AVIP_FLUX_SG;
  SgGeo geo;
  if (use_sg) geo = sg_geometry(dx, dy, 2.0 * Hx, 2.0 * Hy);
#pragma unroll
  for (int s = 0; s < AVIP_MAX_SPECIES; ++s) {
    if (s < ns && !a.ph.sp[s].immobile) {
      const double2* dl = reinterpret_cast<const double2*>(a.ndat + ((size_t)s * a.Npad + lo) * 4);
      const double2* dh = reinterpret_cast<const double2*>(a.ndat + ((size_t)s * a.Npad + hi) * 4);
      const double2 gl = dl[0], vl = dl[1], gh = dh[0], vh = dh[1];
      const EdgeEnd L{n[(size_t)s * a.Npad + lo], gl.x, gl.y, vl.x, vl.y};
      const EdgeEnd H{n[(size_t)s * a.Npad + hi], gh.x, gh.y, vh.x, vh.y};
      a.eflux[(size_t)s * a.E + e] =
          edge_flux(L, H, dx, dy, Hx, Hy, a.ph.sp[s], dt4, a.ph.beta, a.ph.limiter, use_sg ? &geo : nullptr);
    }
  }
}

// Single block: charge in block order, time, parity, statistics; re-arm the dt minimum.
__device__ __forceinline__ void finalize_body(DevScalars* sc, const double* partials, int nparts) {
  __shared__ double sm[32];
  double t = 0.0;
  for (int b = threadIdx.x; b < nparts; b += blockDim.x) t += partials[b];
  const int ln = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (ln == 0) sm[warp] = t;
  __syncthreads();
  if (threadIdx.x == 0) {
    double q = 0.0;
    for (int w = 0; w < nw; ++w) q += sm[w];
    sc->charge = kECharge * q;
    const double dt = sc->dt;
    if (!(dt > 0.0) || !isfinite(dt)) {
      if (sc->status == AVIP_OK) sc->status = AVIP_ENAN;
    }
    sc->t += dt;
    sc->parity ^= 1;
    sc->run_steps += 1;
    sc->run_iters_total += sc->pcg_iters;
    sc->run_iters_max = max(sc->run_iters_max, sc->pcg_iters);
    sc->run_dt_min = fmin(sc->run_dt_min, dt);
    sc->run_dt_max = fmax(sc->run_dt_max, dt);
    sc->run_relres_max = fmax(sc->run_relres_max, sc->pcg_relres);
    sc->dt_bits = (unsigned long long)__double_as_longlong(INFINITY);
  }
}

// Photoionisation (after the Helmholtz solves): S_ph = sum_j S_ph,j added to the electron and
// positive-ion sources, and the chemical time-step limit with the complete electron source.
__global__ void __launch_bounds__(kDDThreads) photo_add_kernel(DDArgs a, int with_dt) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  double chem = INFINITY;
  if (i < a.A.N) {
    double S = 0.0;
    for (int j = 0; j < a.ph.photo_terms; ++j) S += a.photo_psi[(size_t)j * a.Npad + i];
    a.photo_S[i] = S;
    const int ie = a.ph.src_idx[0], ip = a.ph.src_idx[1];
    const double se = a.src[(size_t)ie * a.Npad + i] + S;
    a.src[(size_t)ie * a.Npad + i] = se;
    a.src[(size_t)ip * a.Npad + i] += S;
    if (with_dt && se != 0.0) {
      const double* n = a.nbuf + (size_t)a.sc->parity * AVIP_MAX_SPECIES * a.Npad;
      chem = a.ph.a_chem * fabs(n[(size_t)ie * a.Npad + i]) * recip_nr(fabs(se));
    }
  }
  if (with_dt) block_min_to_global(chem, &a.sc->dt_bits);
}

__global__ void finalize_kernel(DevScalars* sc, const double* partials, int nparts) {
  after_predecessor();
  finalize_body(sc, partials, nparts);
}

__global__ void run_reset_kernel(DevScalars* sc) {
  sc->charge_start = sc->charge;
  sc->run_steps = 0;
  sc->run_iters_total = 0;
  sc->run_iters_max = 0;
  sc->run_dt_min = INFINITY;
  sc->run_dt_max = 0.0;
  sc->run_relres_max = 0.0;
  sc->status = AVIP_OK;
}


// ------------------------------------------------------------------------ FP32 forms
// Mixed precision (ph.dd_fp32): gradients, velocities, sources and fluxes in FP32 with FP32
// accumulation; the density state, the explicit update n += dt (R/V + S), the time-step
// candidates and reduction and the charge sum stay FP64.  Two differences are formed in FP64
// before rounding, because FP32 cannot resolve them from the absolute values: the potential
// differences phi_k - phi_i of the gradient (phi ~ 1e4 V varies by ~10 V between neighbours,
// so E from absolute values would lose 4 digits), using sum_k G_ik = 0 (each cell's nodal
// normals sum to zero), and the edge vectors x_j - x_i (coordinates ~1e-2 m, edges ~1e-5 m).
__device__ __forceinline__ float mobility32(const SpeciesParams& sp, float Emag) {
  if (sp.mob_model == AVIP_MOB_POWER)
    return (float)sp.mob[0] * powf(fmaxf(Emag, (float)sp.mob[3]) / (float)sp.mob[1], (float)sp.mob[2]);
  return (float)sp.mob[0];
}

__device__ __forceinline__ float limiter32(float r, float beta, int kind) {
  if (kind == AVIP_LIM_VANLEER) return (r + fabsf(r)) / (1.0f + fabsf(r));
  return fmaxf(0.0f, fmaxf(fminf(beta * r, 1.0f), fminf(r, beta)));
}

__device__ __forceinline__ void node_fields32_body(const DDArgs& a, int with_dt, int bid) {
  const int i = bid * blockDim.x + threadIdx.x;
  const int N = a.A.N;
  const int ns = a.ph.ns;
  double chem = INFINITY;
  if (i < N) {
    const int slice = i / kSlice, lane = i % kSlice;
    const double* n = a.nbuf + (size_t)a.sc->parity * AVIP_MAX_SPECIES * a.Npad;
    const int base = __ldg(a.A.sl_ptr + slice) + lane;
    const int rl = __ldg(a.A.rlen + i);
    const double phii = a.phi[i];
    float ui[AVIP_MAX_SPECIES];
#pragma unroll
    for (int s = 0; s < AVIP_MAX_SPECIES; ++s) ui[s] = s < ns ? (float)n[(size_t)s * a.Npad + i] : 0.0f;
    float gpx = 0.0f, gpy = 0.0f;
    float gnx[AVIP_MAX_SPECIES], gny[AVIP_MAX_SPECIES];
#pragma unroll
    for (int s = 0; s < AVIP_MAX_SPECIES; ++s) gnx[s] = gny[s] = 0.0f;
    for (int k = 1; k < rl; ++k) {  // slot 0 is the row itself: zero difference
      const int e = base + k * kSlice;
      const int j = __ldg(a.A.col + e);
      const float wx = __ldg(a.gx32 + e), wy = __ldg(a.gy32 + e);
      const float dp = (float)(a.phi[j] - phii);
      gpx = fmaf(wx, dp, gpx);
      gpy = fmaf(wy, dp, gpy);
#pragma unroll
      for (int s = 0; s < AVIP_MAX_SPECIES; ++s) {
        if (s < ns) {
          const float du = (float)n[(size_t)s * a.Npad + j] - ui[s];
          gnx[s] = fmaf(wx, du, gnx[s]);
          gny[s] = fmaf(wy, du, gny[s]);
        }
      }
    }
    const float Ex = -gpx, Ey = -gpy;
    const float Emag = sqrtf(Ex * Ex + Ey * Ey);
    a.Ex[i] = Ex;
    a.Ey[i] = Ey;
    float mu[AVIP_MAX_SPECIES];
#pragma unroll
    for (int s = 0; s < AVIP_MAX_SPECIES; ++s) {
      if (s < ns) {
        const SpeciesParams& sp = a.ph.sp[s];
        mu[s] = mobility32(sp, Emag);
        const float sg = sp.q > 0 ? 1.0f : -1.0f;
        const float vx = sg * mu[s] * Ex, vy = sg * mu[s] * Ey;
        reinterpret_cast<float4*>(a.ndat32)[(size_t)s * a.Npad + i] = make_float4(gnx[s], gny[s], vx, vy);
        const double nmu = n[(size_t)s * a.Npad + i] * (double)mu[s];
        a.nm[(size_t)s * a.Npad + i] = nmu;
        a.vf[(size_t)s * a.Npad + i] = make_float4(vx, vy, (float)nmu, 0.f);
      } else {
        mu[s] = 0.0f;
      }
    }
    float src[AVIP_MAX_SPECIES];
#pragma unroll
    for (int s = 0; s < AVIP_MAX_SPECIES; ++s) src[s] = 0.0f;
    if (a.ph.src_model != AVIP_SRC_NONE) {
      const int ie = a.ph.src_idx[0], ip = a.ph.src_idx[1], ineg = a.ph.src_idx[2];
      const float ne = (float)n[(size_t)ie * a.Npad + i];
      const float alpha = Emag > 0.0f ? (float)a.ph.src_params[0] * expf(-(float)a.ph.src_params[1] / Emag) : 0.0f;
      float mue = 0.0f;
#pragma unroll
      for (int s = 0; s < AVIP_MAX_SPECIES; ++s)
        if (s == ie) mue = mu[s];
      const float ion = alpha * mue * Emag * ne;
#pragma unroll
      for (int s = 0; s < AVIP_MAX_SPECIES; ++s) {
        if (s == ie) src[s] += ion;
        if (s == ip) src[s] += ion;
      }
      if (a.ph.src_model == AVIP_SRC_TOWNSEND_ATTACH) {
        const float att = (float)a.ph.src_params[2] * ne;
#pragma unroll
        for (int s = 0; s < AVIP_MAX_SPECIES; ++s) {
          if (s == ie) src[s] -= att;
          if (s == ineg) src[s] += att;
        }
      } else if (a.ph.src_model == AVIP_SRC_MORROW_LOWKE) {
        float npos = 0.0f, nneg = 0.0f;
#pragma unroll
        for (int s = 0; s < AVIP_MAX_SPECIES; ++s) {
          if (s == ip) npos = (float)n[(size_t)s * a.Npad + i];
          if (s == ineg) nneg = (float)n[(size_t)s * a.Npad + i];
        }
        const float eta =
            Emag > 0.0f ? (float)a.ph.src_params[2] * expf(-(float)a.ph.src_params[3] / Emag) : 0.0f;
        const float att = eta * mue * Emag * ne;
        const float br = (float)a.ph.src_params[4];
        const float rep = br * ne * npos;
        const float rnp = br * nneg * npos;
#pragma unroll
        for (int s = 0; s < AVIP_MAX_SPECIES; ++s) {
          if (s == ie) src[s] = src[s] - att - rep;
          if (s == ip) src[s] = src[s] - rep - rnp;
          if (s == ineg) src[s] = src[s] + att - rnp;
        }
      }
      float se = 0.0f;
#pragma unroll
      for (int s = 0; s < AVIP_MAX_SPECIES; ++s)
        if (s == ie) se = src[s];
      // chemical time-step candidate in FP64 (part of the time-step reduction)
      if (se != 0.0f) chem = a.ph.a_chem * fabs(n[(size_t)ie * a.Npad + i]) / fabs((double)se);
    }
#pragma unroll
    for (int s = 0; s < AVIP_MAX_SPECIES; ++s)
      if (s < ns) a.src[(size_t)s * a.Npad + i] = src[s];
  }
  if (with_dt) block_min_to_global(chem, &a.sc->dt_bits);
}

__global__ void __launch_bounds__(kDDThreads) node_fields32_kernel(DDArgs a, int with_dt) {
  after_predecessor();
  node_fields32_body(a, with_dt, blockIdx.x);
}

struct EdgeEnd32 {
  float u, gx, gy, vx, vy;
};

// FP32 edge flux lo -> hi through (Sx, Sy) oriented lo -> hi; (dx, dy) = x_hi - x_lo.
__device__ __forceinline__ float edge_flux32(const EdgeEnd32& lo, const EdgeEnd32& hi, float dx, float dy, float Sx,
                                             float Sy, float D, float dt, float beta, int lim, int scheme) {
  const float Vx = 0.5f * (lo.vx + hi.vx), Vy = 0.5f * (lo.vy + hi.vy);
  const float gx = 0.5f * (lo.gx + hi.gx), gy = 0.5f * (lo.gy + hi.gy);
  if (scheme == AVIP_FLUX_SG) {
    const float h = sqrtf(dx * dx + dy * dy);
    const float rh = 1.0f / h;
    const float ex = dx * rh, ey = dy * rh;
    const float s = Sx * ex + Sy * ey;
    const float spx = Sx - s * ex, spy = Sy - s * ey;
    const float Vt = Vx * ex + Vy * ey;
    float fpar;
    if (D > 0.0f) {
      const float aa = h * Vt / D, ab = fabsf(aa);
      const float Bp = ab != 0.0f ? ab / expm1f(ab) : 1.0f, Bm = ab + Bp;  // B(|a|), B(-|a|)
      fpar = (D * s * rh) * ((aa >= 0.0f ? Bm : Bp) * lo.u - (aa >= 0.0f ? Bp : Bm) * hi.u);
    } else {
      fpar = s * (fmaxf(Vt, 0.0f) * lo.u + fminf(Vt, 0.0f) * hi.u);
    }
    return fpar + (Vx * spx + Vy * spy) * (0.5f * (lo.u + hi.u)) - D * (gx * spx + gy * spy);
  }
  const float av = Vx * Sx + Vy * Sy;
  const bool up_lo = av >= 0.0f;
  const EdgeEnd32& U = up_lo ? lo : hi;
  const float delta = (up_lo ? hi.u : lo.u) - U.u;
  float psi = 0.0f;
  if (delta != 0.0f) {
    const float ux = up_lo ? dx : -dx, uy = up_lo ? dy : -dy;  // x_W - x_U
    const float r = (2.0f * (U.gx * ux + U.gy * uy) - delta) / delta;
    psi = limiter32(r, beta, lim);
  }
  const float lw = 0.5f * delta - 0.5f * dt * (gx * Vx + gy * Vy);
  return (U.u + lw * psi) * av - D * (gx * Sx + gy * Sy);
}

__device__ __forceinline__ void flux_update32_body(const DDArgs& a, int bid) {
  const int i = bid * blockDim.x + threadIdx.x;
  const int N = a.A.N;
  const int ns = a.ph.ns;
  const double dt = a.ph.dt_fixed > 0.0 ? a.ph.dt_fixed : __longlong_as_double((long long)a.sc->dt_bits);
  const float dtf = (float)dt, betaf = (float)a.ph.beta;
  double qsum = 0.0;
  if (i < N) {
    const int par = a.sc->parity;
    const double* n = a.nbuf + (size_t)par * AVIP_MAX_SPECIES * a.Npad;
    double* nn = a.nbuf + (size_t)(par ^ 1) * AVIP_MAX_SPECIES * a.Npad;
    const float4* nd = reinterpret_cast<const float4*>(a.ndat32);
    const int slice = i / kSlice, lane = i % kSlice;
    const int base = __ldg(a.A.sl_ptr + slice) + lane;
    const int rl = __ldg(a.flen + i);  // edge slots only
    const double xi = a.x[i], yi = a.y[i];
    float R[AVIP_MAX_SPECIES];
    EdgeEnd32 me[AVIP_MAX_SPECIES];
#pragma unroll
    for (int s = 0; s < AVIP_MAX_SPECIES; ++s) {
      R[s] = 0.0f;
      if (s < ns) {
        const float4 d = nd[(size_t)s * a.Npad + i];
        me[s] = EdgeEnd32{(float)n[(size_t)s * a.Npad + i], d.x, d.y, d.z, d.w};
      }
    }
    for (int k = 1; k < rl; ++k) {
      const int e = base + k * kSlice;
      const int j = __ldg(a.A.col + e);
      const float Sx = __ldg(a.sx32 + e), Sy = __ldg(a.sy32 + e);
      const bool lo_is_me = i < j;
      // canonical lo -> hi edge vector, formed in FP64 so that both ends round the same value
      const float dx = lo_is_me ? (float)(a.x[j] - xi) : (float)(xi - a.x[j]);
      const float dy = lo_is_me ? (float)(a.y[j] - yi) : (float)(yi - a.y[j]);
      const float cSx = lo_is_me ? Sx : -Sx, cSy = lo_is_me ? Sy : -Sy;
#pragma unroll
      for (int s = 0; s < AVIP_MAX_SPECIES; ++s) {
        if (s < ns) {
          const float4 d = nd[(size_t)s * a.Npad + j];
          const EdgeEnd32 other{(float)n[(size_t)s * a.Npad + j], d.x, d.y, d.z, d.w};
          const EdgeEnd32& lo = lo_is_me ? me[s] : other;
          const EdgeEnd32& hi = lo_is_me ? other : me[s];
          const float F = edge_flux32(lo, hi, dx, dy, cSx, cSy, (float)a.ph.sp[s].D, dtf, betaf, a.ph.limiter,
                                      a.ph.scheme);
          R[s] = lo_is_me ? R[s] - F : R[s] + F;
        }
      }
    }
    const float Sbx = __ldg(a.sx32 + base), Sby = __ldg(a.sy32 + base);
    const double Vi = a.vol[i];
    bool bad = false;
#pragma unroll
    for (int s = 0; s < AVIP_MAX_SPECIES; ++s) {
      if (s < ns) {
        const SpeciesParams& sp = a.ph.sp[s];
        float Fx = me[s].u * me[s].vx, Fy = me[s].u * me[s].vy;
        if (sp.bnd_mode == AVIP_BND_OUTFLOW) {
          Fx -= (float)sp.D * me[s].gx;
          Fy -= (float)sp.D * me[s].gy;
        }
        const float rs = R[s] - (Fx * Sbx + Fy * Sby);
        // FP64 update of the FP64 state
        const double un = n[(size_t)s * a.Npad + i] + dt * ((double)rs / Vi + a.src[(size_t)s * a.Npad + i]);
        nn[(size_t)s * a.Npad + i] = un;
        bad |= !isfinite(un);
        qsum += sp.q * (Vi * un);
      }
    }
    if (bad) atomicCAS(&a.sc->status, AVIP_OK, AVIP_ENAN);
  }
  block_charge(qsum, a.partials + bid);
  if (bid == 0 && threadIdx.x == 0) a.sc->dt = dt;
}

__global__ void __launch_bounds__(kDDThreads, 3) flux_update32_kernel(DDArgs a) {
  after_predecessor();
  flux_update32_body(a, blockIdx.x);
}

// ------------------------------------------------------------------------ batched forms
// One launch covers every instance of a batch: block b belongs to the instance k with
// bpref[k] <= b < bpref[k + 1] and runs that instance's block b - bpref[k].
__device__ __forceinline__ int batch_instance(const int32_t* __restrict__ bpref, int count, int b) {
  int lo = 0, hi = count;  // largest k with bpref[k] <= b
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (__ldg(bpref + mid) <= b) lo = mid; else hi = mid;
  }
  return lo;
}

__global__ void __launch_bounds__(kDDThreads) node_fields_batch_kernel(const DDArgs* __restrict__ args,
                                                                        const int32_t* __restrict__ bpref, int count) {
  const int k = batch_instance(bpref, count, blockIdx.x);
  const DDArgs& a = args[k];
  if (a.ph.dd_fp32)
    node_fields32_body(a, a.ph.dt_fixed > 0.0 ? 0 : 1, blockIdx.x - __ldg(bpref + k));
  else
    node_fields_body(a, a.ph.dt_fixed > 0.0 ? 0 : 1, blockIdx.x - __ldg(bpref + k));
}
__global__ void __launch_bounds__(kDDThreads) dt_cells_batch_kernel(const DDArgs* __restrict__ args,
                                                                     const int32_t* __restrict__ bpref, int count) {
  const int k = batch_instance(bpref, count, blockIdx.x);
  const DDArgs& a = args[k];
  if (a.ph.dt_fixed > 0.0) return;
  dt_cells_body(a, blockIdx.x - __ldg(bpref + k), __ldg(bpref + k + 1) - __ldg(bpref + k));
}
// (one resident block per SM guaranteed: the per-row evaluation of every edge needs ~140
// registers, and a cap of 128 made it spill)
__global__ void __launch_bounds__(kDDThreads, 1) flux_update_batch_kernel(const DDArgs* __restrict__ args,
                                                                        const int32_t* __restrict__ bpref, int count) {
  const int k = batch_instance(bpref, count, blockIdx.x);
  if (args[k].ph.dd_fp32)
    flux_update32_body(args[k], blockIdx.x - __ldg(bpref + k));
  else
    flux_update_body_t<false>(args[k], blockIdx.x - __ldg(bpref + k));  // batches evaluate each edge per row
}
__global__ void finalize_batch_kernel(const DDArgs* __restrict__ args, int count, int threads) {
  const DDArgs& a = args[blockIdx.x];
  finalize_body(a.sc, a.partials, (a.A.N + threads - 1) / threads);
}
__global__ void run_reset_batch_kernel(const DDArgs* __restrict__ args, int count) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= count) return;
  DevScalars* sc = args[k].sc;
  sc->charge_start = sc->charge;
  sc->run_steps = 0;
  sc->run_iters_total = 0;
  sc->run_iters_max = 0;
  sc->run_dt_min = INFINITY;
  sc->run_dt_max = 0.0;
  sc->run_relres_max = 0.0;
  sc->status = AVIP_OK;
}

// ------------------------------------------------------------------------ host launchers
static inline int nblk(int n) { return (n + kDDThreads - 1) / kDDThreads; }

// Launch with programmatic stream serialisation (see after_predecessor).
template <typename... P, typename... A>
static cudaError_t launch_after(void (*kernel)(P...), int blocks, int threads, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(threads);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

cudaError_t launch_node_fields(const DDArgs& a, int with_dt, cudaStream_t st) {
  return launch_after(a.ph.dd_fp32 ? node_fields32_kernel : node_fields_kernel, nblk(a.A.N), kDDThreads, st, a, with_dt);
}
cudaError_t launch_photo_add(const DDArgs& a, int with_dt, cudaStream_t st) {
  photo_add_kernel<<<nblk(a.A.N), kDDThreads, 0, st>>>(a, with_dt);
  return cudaGetLastError();
}

// Blocks of the cell time step: up to kDtCells cells per thread, one on small meshes (fewer than
// 4 blocks per SM otherwise).
int dt_cells_blocks(int cells, int threads) {
  const int most = (cells + threads - 1) / threads, least = (cells + kDtCells * threads - 1) / (kDtCells * threads);
  return most < 4 * 152 ? most : least < 4 * 152 ? 4 * 152 : least;
}
cudaError_t launch_dt_cells(const DDArgs& a, cudaStream_t st) {
  const int blocks = dt_cells_blocks(a.T, kDDThreads);
  return launch_after(dt_cells_kernel, blocks, kDDThreads, st, a);
}
cudaError_t launch_flux_update(const DDArgs& a, cudaStream_t st) {
  if (a.ph.dd_fp32) return launch_after(flux_update32_kernel, nblk(a.A.N), kDDThreads, st, a);
  if (!(a.eflux && a.E > 0)) return launch_after(flux_update_kernel<false>, nblk(a.A.N), kDDThreads, st, a);
  const cudaError_t e = launch_after(edge_flux_kernel, nblk(a.E), kDDThreads, st, a);
  return e != cudaSuccess ? e : launch_after(flux_update_kernel<true>, nblk(a.A.N), kDDThreads, st, a);
}
cudaError_t launch_finalize(DevScalars* sc, const double* partials, int nparts, cudaStream_t st) {
  return launch_after(finalize_kernel, 1, 256, st, sc, partials, nparts);
}
cudaError_t launch_run_reset(DevScalars* sc, cudaStream_t st) {
  run_reset_kernel<<<1, 1, 0, st>>>(sc);
  return cudaGetLastError();
}
// ------------------------------------------------------------------ checkpoint copies
// state_get: the device state in the caller's layout (one coalesced read per field, a scattered
// write to the caller positions); state_put: the reverse, after state_check has found every
// entry finite.  Values are copied, never recomputed, so a checkpoint round trip is exact.
__global__ void state_take_kernel(StateArgs s) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const size_t N = (size_t)s.N;
  const size_t hb = (size_t)(s.ns + 1) * N + 1;  // first predictor-history entry
  if (i == 0) {
    s.stage[(size_t)(s.ns + 1) * N] = s.sc->t;
    s.stage[hb + 3 * N] = (double)s.sc->phi_hist;
  }
  if (i >= s.N) return;
  const size_t c = (size_t)__ldg(s.perm + i);
  const double* n = s.nbuf + (size_t)s.sc->parity * AVIP_MAX_SPECIES * s.Npad;
  for (int k = 0; k < s.ns; ++k) s.stage[k * N + c] = n[(size_t)k * s.Npad + i];
  s.stage[s.ns * N + c] = s.phi[i];
  s.stage[hb + c] = s.phi1[i];
  s.stage[hb + N + c] = s.phi2[i];
  s.stage[hb + 2 * N + c] = s.phi3[i];
}
__global__ void state_check_kernel(StateArgs s) {
  const size_t total = (size_t)(s.ns + 4) * s.N + 2;
  bool bad = false;
  for (size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x; k < total; k += (size_t)gridDim.x * blockDim.x)
    bad |= !isfinite(s.stage[k]);
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicExch(s.flag, 1);
}
__global__ void state_put_kernel(StateArgs s) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const size_t N = (size_t)s.N;
  const size_t hb = (size_t)(s.ns + 1) * N + 1;
  if (i == 0) {
    s.sc->t = s.t;
    s.sc->phi_hist = s.hist;
  }
  if (i >= s.N) return;
  const size_t c = (size_t)__ldg(s.perm + i);
  double* n = s.nbuf + (size_t)s.sc->parity * AVIP_MAX_SPECIES * s.Npad;
  for (int k = 0; k < s.ns; ++k) n[(size_t)k * s.Npad + i] = s.stage[k * N + c];
  s.phi[i] = s.stage[s.ns * N + c];
  s.phi1[i] = s.stage[hb + c];
  s.phi2[i] = s.stage[hb + N + c];
  s.phi3[i] = s.stage[hb + 2 * N + c];
}
cudaError_t launch_state_take(const StateArgs& s, cudaStream_t st) {
  state_take_kernel<<<nblk(s.N), kDDThreads, 0, st>>>(s);
  return cudaGetLastError();
}
cudaError_t launch_state_check(const StateArgs& s, cudaStream_t st) {
  state_check_kernel<<<nblk(s.N), kDDThreads, 0, st>>>(s);
  return cudaGetLastError();
}
cudaError_t launch_state_put(const StateArgs& s, cudaStream_t st) {
  state_put_kernel<<<nblk(s.N), kDDThreads, 0, st>>>(s);
  return cudaGetLastError();
}

int flux_blocks(int N) { return nblk(N); }
// Charge partials a handle must hold: one per block at the smallest batched block size.
int flux_partials_max(int N) { return (N + kDDMinThreads - 1) / kDDMinThreads; }

// The drift-diffusion stages of a batch with `threads` threads per block (kDDMinThreads ..
// kDDThreads, a multiple of 32; the block prefix sums node_pref / cell_pref were made for it).
cudaError_t launch_dd_batch(const DDArgs* args, const int32_t* node_pref, const int32_t* cell_pref, int count,
                            int node_blocks, int cell_blocks, int threads, cudaStream_t st) {
  if (threads < kDDMinThreads || threads > kDDThreads || threads % 32) return cudaErrorInvalidValue;
  node_fields_batch_kernel<<<node_blocks, threads, 0, st>>>(args, node_pref, count);
  dt_cells_batch_kernel<<<cell_blocks, threads, 0, st>>>(args, cell_pref, count);
  flux_update_batch_kernel<<<node_blocks, threads, 0, st>>>(args, node_pref, count);
  finalize_batch_kernel<<<count, 256, 0, st>>>(args, count, threads);
  return cudaGetLastError();
}
cudaError_t launch_run_reset_batch(const DDArgs* args, int count, cudaStream_t st) {
  run_reset_batch_kernel<<<(count + 127) / 128, 128, 0, st>>>(args, count);
  return cudaGetLastError();
}
int dd_threads() { return kDDThreads; }

}  // namespace avip
