// FP64 Picard predictor (Eq. (5)) of the nonlinear conservative systems with its contractions on the
// integer pipe (fx.cuh).
//
// The FP64 pipe (2 lane operations per clock and SM) is what bounds the predictor, and nine tenths
// of its FP64 work are products: with the fixed 1-D tables (the derivative along each direction,
// the time solve, the time averages, the weak form and the face values) and of the flux itself.
// Here FP64 forms 1/rho, the velocities and the pressure once per node; velocities, momenta,
// p and H = E + p are then 64-bit fixed-point numbers, a flux component is one integer product
// (momentum or H times velocity, + p), and every line of n of them is contracted in fixed point.
// The directions are summed as integers, the time solve takes the sums as they are, and one FP64
// FMA per value forms q = u + dt Kw R.  From the constant guess the first iteration has one time
// level, q^0 = u, so its right-hand side is formed once.
//
// Scale: one power of two per cell and quantity, one to two bits above its largest magnitude at
// u^n: velocities s = |v| + c, momenta rho s, H (shallow water: s, h s, and the larger of |h + b| and
// h for the surface); a flux has the product's scale.  An iterate above it, a non-finite value or magnitudes
// outside 2^-100 .. 2^100 end the attempt, and the cell is recomputed by the FP64 form
// (predictor_cell), whose results for such values are kept as they were.  A contraction's rounding
// is 2^-58 of the scale times the table's row sum: below the rounding of the FP64 FMA chain,
// which starts from fluxes rounded at 2^-53.
//
// Work split: a task is one line (time level, transverse node, variable) of one direction, so each
// flux value is formed once and used n times from registers; results are added to the integer
// sums in shared memory, direction by direction (no two tasks of a direction share a result).
// Tasks run over the variables fastest: neighbouring lanes read neighbouring words of the
// [node][variable] records.  Three blocks of 10 warps an SM at 3-D order 4 (64 registers, some
// spilled): the phases of one block, FP64 or integer, overlap the others' (two blocks of 96
// registers: 18 % slower).
//
// Measured, one step, predictor alone, against the FP64 form: 3-D Euler order 4, 32^3 cells 33.0 ->
// 7.6 ms; order 3, 40^3 18.8 -> 4.7 ms; shallow water order 3, 768^2 34.4 -> 9.5 ms (FP64 pipe 50 %
// busy, issue slots 50 %, barriers and latency the rest).  Error of a step against binary64 as
// before, 1.6e-16 of the state at 3-D order 4, 2.5e-16 (2.4e-16) for shallow water.
#pragma once
#include "fx.cuh"
#include "kernels.cuh"

namespace ader {

// Scales of a cell's fixed-point quantities.
struct FxScale {
  int v, j, H, s;  // velocities, momenta, H, shallow water's surface
};

// Node records of the fixed-point form, in place of the state's: Euler (p, j[D], H) in the scales
// (momentum flux, j, H); shallow water (h + b, hu, hv, g h as a double).  The velocities, as
// fractions v 2^(1084 - E.v) < 2^62, are in their own array V[node][D].  Factors are kept split.
template <class P, int D, int N>
struct FxCell {
  using C = Cfg<P, D, N>;
  static constexpr bool EULER = !P::NCPS;
  static constexpr int NV = C::NV, NVF = EULER ? NV : NV - 1;  // variables with a flux (b has none)

  // scale of variable v's flux (shallow water, v = 3: the surface)
  __device__ static int flux_scale(const FxScale& E, int v) {
    if (v == 0) return E.j;
    if (v == NV - 1) return EULER ? E.H + E.v - 1020 : E.s;
    return E.j + E.v - 1020;
  }
  // F_d[v] of a node in that scale, split (shallow water, v = 3: the surface); below 2^60
  template <int d>
  __device__ static fx2 flux(const fx2* rec, const fx2* V, int node, int v) {
    const fx2* r = rec + node * NV;
    const fx2 a = r[v == 0 ? 1 + d : (!EULER && v == 3 ? 0 : v)];
    if (v == 0 || (!EULER && v == 3)) return a;
    long long f = fx_mul(a, V[node * D + d]);
    if (EULER && v == 1 + d) f += *reinterpret_cast<const long long*>(r);
    return fx_split(f);
  }
};

// 1/x for a normal x: a 20-bit approximation and one step of the cubic (Halley) iteration,
// r (1 + e + e^2) with e = 1 - x r.  Zero, infinite and NaN x give a non-finite or zero r (the
// scale's tests follow).
__device__ __forceinline__ double fx_rcp(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

template <int D>
__device__ __forceinline__ void fx_velocities(const double* q, double (&v)[D]) {
  const double ir = fx_rcp(q[0]);
#pragma unroll
  for (int i = 0; i < D; ++i) v[i] = q[1 + i] * ir;
}

template <int D>
__device__ __forceinline__ double fx_pressure(const PdeParams& pp, const double* q,
                                              const double (&v)[D]) {
  double jv = 0.0;
#pragma unroll
  for (int i = 0; i < D; ++i) jv = fma(q[1 + i], v[i], jv);
  return (pp.gamma - 1.0) * fma(-0.5, jv, q[D + 1]);
}

// State records of nt time levels -> fixed-point records and velocities.
template <class P, int D, int N>
__device__ __forceinline__ void fx_nodes(const PdeParams& pp, double* q, fx2* V,
                                         const FxScale& E, int nt, int& over, int tid) {
  using C = Cfg<P, D, N>;
  using X = FxCell<P, D, N>;
  for (int k = tid; k < nt * C::NS; k += C::TPB) {
    double* qn = q + k * C::NV;
    fx2* rn = reinterpret_cast<fx2*>(qn);
    double v[D];
    fx_velocities<D>(qn, v);
#pragma unroll
    for (int i = 0; i < D; ++i) V[k * D + i] = fx_split(fx_in<9>(v[i], E.v, over));
    if constexpr (X::EULER) {
      const double p = fx_pressure<D>(pp, qn, v);
      rn[D + 1] = fx_split(fx_in(qn[D + 1] + p, E.H, over));
      // the products are below 2^58, and p is kept below it
      *reinterpret_cast<long long*>(rn) = fx_in<5>(p, E.j + E.v - 1022, over);
    } else {
      const double h = qn[0];
      rn[0] = fx_split(fx_in(h + qn[3], E.s, over));
      qn[3] = pp.grav * h;
    }
#pragma unroll
    for (int i = 0; i < D; ++i) rn[1 + i] = fx_split(fx_in(qn[1 + i], E.j, over));
  }
}

// Scales from the largest magnitudes of the state u (level 0 of q) over the cell; false when one is
// outside 2^-100 .. 2^100 or not finite.  s_mag: three words of shared memory, zeroed.
template <class P, int D, int N>
__device__ __forceinline__ bool fx_scales(const PdeParams& pp, const double* q, unsigned* s_mag,
                                          FxScale& E, int tid) {
  using C = Cfg<P, D, N>;
  using X = FxCell<P, D, N>;
  unsigned m[3] = {0u, 0u, 0u};  // Euler rho, H, s; shallow water h, max(|h + b|, h), s
  for (int k = tid; k < C::NS; k += C::TPB) {
    const double* qn = q + k * C::NV;
    double v[D];
    fx_velocities<D>(qn, v);
    float x[3], vm = 0.f;
#pragma unroll
    for (int i = 0; i < D; ++i) vm += fabsf(__double2float_rn(v[i]));
    x[0] = __double2float_rn(qn[0]);
    if constexpr (X::EULER) {
      const double p = fx_pressure<D>(pp, qn, v);
      x[1] = __double2float_rn(qn[D + 1] + p);
      x[2] = vm + sqrtf(fabsf((float)pp.gamma * __double2float_rn(p) / x[0]));
    } else {
      x[1] = __double2float_rn(qn[0] + qn[3]);
      x[2] = vm + sqrtf((float)pp.grav * fabsf(x[0]));
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const unsigned b = __float_as_uint(x[i]) & 0x7fffffffu;  // NaN and infinity are the largest
      m[i] = b > m[i] ? b : m[i];
    }
  }
  // the surface may lie at the datum (still water with b = -h), and leave it by any factor in a step;
  // h and b are rounded at 2^-53 of h themselves.  Water at rest, 256^2 cells, order 3: 4.0 ms in the
  // FP64 form, 1.2 here.
  if (!X::EULER && m[0] > m[1]) m[1] = m[0];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const unsigned w = __reduce_max_sync(0xffffffffu, m[i]);
    if ((tid & 31) == 0) atomicMax(&s_mag[i], w);
  }
  __syncthreads();
  bool fit = true;
  int ex[3];
  float mt[3];  // magnitude = mt 2^ex, 1 <= mt < 2
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const unsigned b = s_mag[i];
    fit = fit && b > 0x0d800000u && b < 0x71800000u;
    ex[i] = (int)(b >> 23) - 127;
    mt[i] = __uint_as_float((b & 0x7fffffu) | 0x3f800000u);
  }
  // the exponent above the magnitude; one bit of room for the iterates' momenta, H and surface (the
  // velocities' is in s, which has the sound speed)
  E.v = ex[2] + 1 + 1022;
  E.j = ex[0] + ex[2] + (mt[0] * mt[2] >= 1.999f ? 2 : 1) + 1 + 1022;
  E.H = ex[1] + 1 + 1 + 1022;
  E.s = ex[1] + 1 + 1 + 1022;
  return fit;
}

// Lines of direction d: R[t][j][v] (+)= sum_m D[j_d][m] F_d[v](t, j_d -> m) for nt time levels
// (shallow water: v = 3 is the surface's derivative, to G[d][t][j]).
template <class P, int D, int N, int d>
__device__ __forceinline__ void fx_lines(const TablesX& TX, const fx2* rec,
                                         const fx2* V, long long* R, long long* G, int nt,
                                         int tid) {
  using C = Cfg<P, D, N>;
  using X = FxCell<P, D, N>;
  constexpr int n = C::n, NV = C::NV, NL = C::NL, NS = C::NS, NF = C::NF;
  constexpr int st = ipow(n, d);
  for (int k = tid; k < nt * NF * NV; k += C::TPB) {
    const int ln = k / NV, v = k - ln * NV;
    const int t = ln / NF, jp = ln - t * NF;
    const int j0 = (jp % st) + (jp / st) * st * n;
    fx2 x[n];
#pragma unroll
    for (int m = 0; m < n; ++m) x[m] = X::template flux<d>(rec, V, t * NS + j0 + m * st, v);
    const bool surf = P::NCPS && v == 3;
    long long* r = surf ? G + d * C::NST + t * NS + j0 : R + t * NL + j0 * NV + v;
    const int sr = surf ? st : st * NV;
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const long long f = fx_dot<n, FX_SHD, false>(x, TX.D[d][i]);
      r[i * sr] = d == 0 || surf ? f : r[i * sr] + f;
    }
  }
}

// Sums R of nt time levels of q, all directions: the state records become fixed-point records.
// Starts after and ends with a barrier.
template <class P, int D, int N>
__device__ __forceinline__ void fx_rhs(const StepArgs& A, const TablesX& TX, double* q, fx2* V,
                                       long long* R, long long* G, const FxScale& E, int nt,
                                       int& over, int tid) {
  using C = Cfg<P, D, N>;
  const fx2* rec = reinterpret_cast<const fx2*>(q);
  fx_nodes<P, D, N>(A.p, q, V, E, nt, over, tid);
  __syncthreads();
  fx_lines<P, D, N, 0>(TX, rec, V, R, G, nt, tid);
  __syncthreads();
  fx_lines<P, D, N, 1>(TX, rec, V, R, G, nt, tid);
  __syncthreads();
  if constexpr (D == 3) {
    fx_lines<P, D, N, 2>(TX, rec, V, R, G, nt, tid);
    __syncthreads();
  }
  if constexpr (P::NCPS) {
    // the node's own g h times the surface derivatives, on the momenta (in the units of R, < 2^58)
    const int km = E.j + E.v - 1020 + TX.kR + 1080;
    for (int k = tid; k < nt * C::NS; k += C::TPB) {
      const double gh = q[k * C::NV + 3];
#pragma unroll
      for (int d = 0; d < D; ++d) {
        const double g = fx_out(G[d * C::NST + k], E.s + TX.kR);
        R[k * C::NV + 1 + d] += fx_in<5>(gh * g, km, over);
      }
    }
    __syncthreads();
  }
}

// One cell; false (for every thread of the block) when a magnitude leaves the scale.
template <class P, int D, int N>
__device__ __forceinline__ bool predictor_cell_fx(const StepArgs& A, const Tables& T,
                                                  const TablesX& TX, long long c) {
  using C = Cfg<P, D, N>;
  using X = FxCell<P, D, N>;
  constexpr int n = C::n, NV = C::NV, NL = C::NL, NS = C::NS, TPB = C::TPB, LPT = C::LPT;
  constexpr int NF = C::NF, FR = C::FR;
  extern __shared__ double smem[];
  double* q = smem;                                              // [n][NL]
  fx2* V = reinterpret_cast<fx2*>(q + n * NL);                    // [NST][D]
  long long* R = reinterpret_cast<long long*>(V + C::NST * D);   // [n][NL]
  long long* G = R + C::FSLOTS * NL;  // [D][NST] surface derivatives (shallow water)
  __shared__ unsigned s_mag[3];
  __shared__ double sdt[n];  // dt x_t times -max 1/h
  const int tid = threadIdx.x;
  const double dt = A.dev->dt;
  const double dm = dt * TX.mih;
  const double* u = A.u + c * NL;
  if (tid < 3) s_mag[tid] = 0u;
  if (tid < n) sdt[tid] = dm * T.x[tid];
  double ul[LPT];
#pragma unroll
  for (int k = 0; k < LPT; ++k) {
    const int l = tid + k * TPB;
    ul[k] = 0.0;
    if (l < NL) q[l] = ul[k] = u[l];
  }
  __syncthreads();
  FxScale E;
  if (!fx_scales<P, D, N>(A.p, q, s_mag, E, tid)) return false;
  int over = 0;
  if (A.cerk) {
    // Runge-Kutta guess (see cerk_guess_cell): the stages on time level 0
    double ks[4][LPT];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (i > 0) {
#pragma unroll
        for (int k = 0; k < LPT; ++k) {
          const int l = tid + k * TPB;
          if (l < NL) q[l] = fma((i == 3 ? 1.0 : 0.5) * dt, ks[i > 0 ? i - 1 : 0][k], ul[k]);
        }
        __syncthreads();
      }
      fx_rhs<P, D, N>(A, TX, q, V, R, G, E, 1, over, tid);
#pragma unroll
      for (int k = 0; k < LPT; ++k) {
        const int l = tid + k * TPB, v = l % NV;
        ks[i][k] = 0.0;
        if (l < NL && v < X::NVF) ks[i][k] = TX.mih * fx_out(R[l], X::flux_scale(E, v) + TX.kR);
      }
    }
    if (__syncthreads_or(over < 0)) return false;
#pragma unroll
    for (int k = 0; k < LPT; ++k) {
      const int l = tid + k * TPB;
      if (l < NL) {
#pragma unroll
        for (int t = 0; t < n; ++t)
          q[t * NL + l] = ul[k] + dt * (T.cerk[0][t] * ks[0][k] + T.cerk[1][t] * (ks[1][k] + ks[2][k]) +
                                        T.cerk[2][t] * ks[3][k]);
      }
    }
  } else {
    // first iteration from q^0 = u: one right-hand side for every time level
    fx_rhs<P, D, N>(A, TX, q, V, R, G, E, 1, over, tid);
    if (__syncthreads_or(over < 0)) return false;
#pragma unroll
    for (int k = 0; k < LPT; ++k) {
      const int l = tid + k * TPB, v = l % NV;
      if (l < NL) {
        const double r = v < X::NVF ? fx_out(R[l], X::flux_scale(E, v) + TX.kR) : 0.0;
#pragma unroll
        for (int t = 0; t < n; ++t) q[t * NL + l] = fma(sdt[t], r, ul[k]);
      }
    }
  }
  __syncthreads();
  for (int it = A.cerk ? 0 : 1; it < A.iters; ++it) {
    fx_rhs<P, D, N>(A, TX, q, V, R, G, E, n, over, tid);
    if (__syncthreads_or(over < 0)) return false;
#pragma unroll
    for (int k = 0; k < LPT; ++k) {
      const int l = tid + k * TPB, v = l % NV;
      if (l < NL) {
        if (v < X::NVF) {
          fx2 x[n];
#pragma unroll
          for (int m = 0; m < n; ++m) x[m] = fx_split(R[m * NL + l]);
          const int ke = X::flux_scale(E, v) + TX.kS;
#pragma unroll
          for (int t = 0; t < n; ++t) q[t * NL + l] = fma(dm, fx_out(fx_dot<n, FX_SHK>(x, TX.Kw[t]), ke), ul[k]);
        } else {
#pragma unroll
          for (int t = 0; t < n; ++t) q[t * NL + l] = ul[k];
        }
      }
    }
    __syncthreads();
  }

  // ---- epilogue: time averages of q (FP64) and of F_d (fixed point) at the owned values ---------
  double* qb = reinterpret_cast<double*>(R);  // [NL]
  long long* FB = R + NL;                     // [D][NL]
#pragma unroll
  for (int k = 0; k < LPT; ++k) {
    const int l = tid + k * TPB;
    if (l < NL) {
      double a = 0.0;
#pragma unroll
      for (int t = 0; t < n; ++t) a = fma(T.w[t], q[t * NL + l], a);
      qb[l] = a;
    }
  }
  __syncthreads();
  const fx2* rec = reinterpret_cast<const fx2*>(q);
  fx_nodes<P, D, N>(A.p, q, V, E, n, over, tid);
  if (__syncthreads_or(over < 0)) return false;
  if constexpr (P::NCPS) {
    // derivatives of the final predictor's surface: lines (direction, time level, transverse node)
    for (int k = tid; k < D * n * NF; k += TPB) {
      const int d = k / (n * NF), t = (k / NF) % n, jp = k % NF;
      const int st = d == 0 ? 1 : n, j0 = d == 0 ? jp * n : jp;
      fx2 x[n];
#pragma unroll
      for (int m = 0; m < n; ++m) x[m] = rec[(t * NS + j0 + m * st) * NV];
#pragma unroll
      for (int i = 0; i < n; ++i)
        G[d * C::NST + t * NS + j0 + i * st] = d == 0 ? fx_dot<n, FX_SHD, false>(x, TX.D[0][i]) : fx_dot<n, FX_SHD, false>(x, TX.D[1][i]);
    }
  }
#pragma unroll
  for (int k = 0; k < LPT; ++k) {
    const int l = tid + k * TPB;
    if (l < NL) {
      const int j = l / NV, v = l - j * NV;
      if (v < X::NVF) {
        fx2 x[n];
#pragma unroll
        for (int t = 0; t < n; ++t) x[t] = X::template flux<0>(rec, V, t * NS + j, v);
        FB[l] = fx_dot<n, FX_SHW>(x, TX.w);
#pragma unroll
        for (int t = 0; t < n; ++t) x[t] = X::template flux<1>(rec, V, t * NS + j, v);
        FB[NL + l] = fx_dot<n, FX_SHW>(x, TX.w);
        if constexpr (D == 3) {
#pragma unroll
          for (int t = 0; t < n; ++t) x[t] = X::template flux<2>(rec, V, t * NS + j, v);
          FB[2 * NL + l] = fx_dot<n, FX_SHW>(x, TX.w);
        }
      } else {
#pragma unroll
        for (int d = 0; d < D; ++d) FB[d * NL + l] = 0;
      }
    }
  }
  __syncthreads();

  // ---- lines of the averages, direction by direction: the face records (q and F_d extrapolated to
  // both ends), and the volume term with the cell-local part of the face terms, from the face
  // fluxes as recorded (the corrector takes off the same values), summed in the velocities' place
  long long* S = reinterpret_cast<long long*>(V);  // [NL]: NST D words hold NL (n D >= NV)
  static_assert(n * D >= NV, "room for the volume sums");
  double* fc = A.face + c * (long long)(D * 2 * FR);
  // FB is in the units 2^(E + kw): inputs of scale E + kw + 1082 for its own contractions
  const int kb = TX.kw + 1082;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const int st = (d == 0 ? 1 : (d == 1 ? n : n * n));
    for (int k = tid; k < NF * NV; k += TPB) {
      const int v = k % NV, jp = k / NV;
      const int j0 = (jp % st) + (jp / st) * st * n;
      const int Eb = X::flux_scale(E, v) + kb;
      fx2 x[n + 2], y[n];
      double q0 = 0.0, q1 = 0.0;
#pragma unroll
      for (int m = 0; m < n; ++m) {
        const int l = (j0 + m * st) * NV + v;
        x[m] = y[m] = fx_split(FB[d * NL + l]);
        q0 = fma(T.e0[m], qb[l], q0);
        q1 = fma(T.e1[m], qb[l], q1);
      }
      const double f0 = fx_out(fx_dot<n, FX_SHK>(y, TX.e[0]), Eb + TX.ke);
      const double f1 = fx_out(fx_dot<n, FX_SHK>(y, TX.e[1]), Eb + TX.ke);
      double* r = fc + d * 2 * FR + k;
      r[0] = q0;
      r[FR] = q1;
      r[NF * NV] = f0;
      r[FR + NF * NV] = f1;
      x[n] = fx_split(fx_in(f0, Eb, over));
      x[n + 1] = fx_split(fx_in(f1, Eb, over));
#pragma unroll
      for (int i = 0; i < n; ++i) {
        long long* s = S + (j0 + i * st) * NV + v;
        const long long f = fx_dot<n + 2, FX_SHS>(x, TX.S[d][i]);
        *s = d == 0 ? f : *s + f;
      }
    }
    if (__syncthreads_or(over < 0)) return false;  // (the FP64 form writes the records again)
  }
  double* un = A.u_next + c * NL;
#pragma unroll
  for (int k = 0; k < LPT; ++k) {
    const int l = tid + k * TPB;
    if (l < NL) {
      const int j = l / NV, v = l - j * NV;
      double s = v < X::NVF ? fx_out(S[l], X::flux_scale(E, v) + kb + TX.kV) : 0.0;
      if constexpr (P::NCPS) {
        // time average of the state-dependent product taken node by node
        if (v == 1 || v == 2) {
          double nb = 0.0;
#pragma unroll
          for (int t = 0; t < n; ++t)
            nb = fma(T.w[t] * q[(t * NS + j) * NV + 3], fx_out(G[(v - 1) * C::NST + t * NS + j], E.s + TX.kR), nb);
          s -= nb;
        }
      }
      un[l] = fma(-dm, s, ul[k]);
    }
  }
  return true;
}

// The FP64 form as the way out of the scale (not inlined: its registers do not add to the integer
// form's).
template <class P, int D, int N>
__device__ __noinline__ void predictor_cell_plain(const StepArgs& A, const Tables& T, long long c) {
  __syncthreads();
  predictor_cell<P, D, N>(A, T, c);
}

template <class P, int D, int N>
__global__ void __launch_bounds__(Cfg<P, D, N>::TPB, Cfg<P, D, N>::MINB)
    k_predictor_fx(const __grid_constant__ StepArgs A, const __grid_constant__ Tables T,
                   const __grid_constant__ TablesX TX) {
  if (A.skip && A.skip[blockIdx.x]) return;  // computes with FV in this step
  if (!predictor_cell_fx<P, D, N>(A, T, TX, blockIdx.x)) predictor_cell_plain<P, D, N>(A, T, blockIdx.x);
}

}  // namespace ader
