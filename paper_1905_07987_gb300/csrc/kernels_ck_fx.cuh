// Elastic predictors (Cauchy-Kowalevski and Picard) with their arithmetic in 64-bit block fixed point
// on the integer pipe (fx.cuh).
//
// The FP64 form (predictor_ck_block) keeps the FP64 pipe 94 % busy: 132 FMAs per node and level at
// order 5, at 2 lane operations per clock and SM.  Here the cell's state is converted once, and
// the levels b_{k+1} = r_k dt L b_k, b_0 = u, whose sum is the time average qbar (r_k: ratios of the
// Taylor or Picard weights), L qbar and the face values are integer arithmetic; FP64 adds the
// update to u once per value.
//
// Parity basis: along each direction a field is kept as sums and differences of mirrored nodes.
// The Gauss-Legendre derivative matrix takes even parts to odd ones and odd to even, so a line of n
// costs n^2 / 2 products in place of n^2 (18 in place of 36 at order 5); the material products and
// the sum over the levels commute with the change of basis, which is paid once on the way in and
// out (24 additions per octet of nodes).
//
// Scale: one power of two per cell, velocities and stresses related by the power of two nearest
// the impedance rho vp: nodal values below 2^57, parity values (sums of eight) below 2^60.  The
// levels shrink at stable time steps; a value that leaves 2^60, a coefficient that does not fit, a
// non-finite value, a cell of values near an end of binary64's range (all below 2^-722, but not all
// zero), and the cell with the point source send the block to the FP64 form.  Rounding:
// 2^-57 of the cell's largest value in the conversion, less in each level (every product takes its
// low words too), where FP64 rounds each operation at 2^-53.
//
// One thread per node, slots of n^3 threads per cell.  Per level two phases: a thread per line
// (18 variable-direction pairs x n^2 lines: n loads, n results), then a thread per node for the
// material products of its 18 derivatives.  Shared memory per cell: the current level and the
// derivatives, split into words, 27 n^3 of them; 28 warps an SM at 72 registers (21 warps: 5 %
// slower, 35 with more spills: 3 %).
//
// Measured, one step, the predictor alone, against the FP64 form, 40^3 cells at order 5: 24.0 -> 5.5
// ms (multiply pipe and issue: 50 % of the issue slots), order 4: 11.4 -> 2.6 ms.  Error of a step
// against binary64: 1.6e-16 .. 4.7e-16 of the state at orders 1 to 5, as before within 7 %.
#pragma once
#include "fx.cuh"
#include "kernels_ck.cuh"

namespace ader {

template <int N>
struct CfgE {
  static constexpr int n = N + 1, NS = n * n * n, NV = 9, NL = NS * NV, NF = n * n;
  static constexpr int H = n / 2, M = (n + 1) / 2;     // mirrored pairs; with the middle
  static constexpr bool ODD = n % 2 != 0;
  static constexpr int NSP = NS | 1;                   // odd stride between variables
  static constexpr int CPB = ck_cells_per_block(N);
  static constexpr int TPB = (CPB * NS + 31) / 32 * 32;
  static constexpr size_t CELL = ((size_t)27 * NSP * sizeof(fx2) + 15) / 16 * 16;
  static constexpr size_t SMEM_X = CPB * (CELL + (fxe_levels(N) + 1) * 12 * sizeof(fx2));
  static constexpr size_t SMEM = SMEM_X > CfgCK<N>::SMEM ? SMEM_X : CfgCK<N>::SMEM;
  static constexpr int MINB = 896 / TPB;  // 28 warps per SM
};

__device__ __forceinline__ long long fx_join(fx2 a) { return ((long long)a.h << 32) + a.l; }

// Parity butterflies of an octet x[z][y][x] of mirrored nodes (forward and, but for the factor 8,
// inverse): along each direction (a, b) -> (a + b, a - b).
__device__ __forceinline__ void fx_octet(long long (&x)[8]) {
#pragma unroll
  for (int s = 1; s < 8; s <<= 1)
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (!(i & s)) {
        const long long a = x[i], b = x[i | s];
        x[i] = a + b;
        x[i | s] = a - b;
      }
}

// Negative when a cell's values, all small, are not all zero (or subnormal): a quiet cell stays.
static __device__ __noinline__ int fxe_tiny(const double* x, int j, int n, int step) {
  int t = 0;
  for (int r = j; r < n; r += step) t |= __double2hiint(x[r]) & 0x7ff00000;
  return -t;
}

// The lines of thread j of a cell, the same in every level: place of the first node in the level (12
// bits) and in the derivatives (13 bits) and the direction; -1: none.  Line id: q = 6 d + i (direction,
// i-th of its six variables: the velocities, then sigma_{0d}, sigma_{1d}, sigma_{2d}).
template <int N>
struct FxeLines {
  using C = CfgE<N>;
  static constexpr int RND = (18 * C::NF + C::NS - 1) / C::NS;
  int t[RND];
  __device__ __forceinline__ explicit FxeLines(int j) {
    constexpr int n = C::n, NF = C::NF;
#pragma unroll
    for (int k = 0; k < RND; ++k) {
      const int id = j + k * C::NS, q = id / NF;
      const int ln = id - q * NF, d = q / 6, i = q - d * 6, b = i - 3;
      const int v = i < 3 ? i : (b == d ? 3 + d : 5 + b + d);
      const int j0 = d == 0 ? ln * n : (d == 1 ? ln % n + (ln / n) * n * n : ln);
      t[k] = id < 18 * NF ? (v * C::NSP + j0) | (q * C::NSP + j0) << 12 | d << 25 : -1;
    }
  }
  // line k: places and stride
  __device__ __forceinline__ bool get(int k, int& x, int& g, int& st) const {
    constexpr int n = C::n;
    x = t[k] & 0xfff;
    g = (t[k] >> 12) & 0x1fff;
    const int d = t[k] >> 25;
    st = d == 0 ? 1 : (d == 1 ? n : n * n);
    return t[k] >= 0;
  }
  static_assert(9 * C::NSP <= 4096 && 18 * C::NSP <= 8192, "places fit their bits");
};

// One application of r dt L to the level X: derivatives of every line into G.
template <int N>
__device__ __forceinline__ void fxe_lines(const TablesE& E, const fx2* X, fx2* G, const FxeLines<N>& L) {
  using C = CfgE<N>;
  constexpr int n = C::n, H = C::H;
#pragma unroll
  for (int r = 0; r < FxeLines<N>::RND; ++r) {
    int px, pg, st;
    if (!L.get(r, px, pg, st)) continue;
    const fx2* x = X + px;
    fx2* g = G + pg;
    fx2 a[n];
#pragma unroll
    for (int m = 0; m < n; ++m) a[m] = x[m * st];
#pragma unroll
    for (int k = 0; k < H; ++k) {
      FxAcc<FXE_SHG> ev, od;
#pragma unroll
      for (int m = 0; m < H; ++m) {
        ev.mac(a[n - 1 - m], E.ev[k][m]);
        od.mac(a[m], E.od[k][m]);
      }
      if (C::ODD) od.mac(a[H], E.od[k][H]);
      g[k * st] = fx_split(ev.get());
      g[(n - 1 - k) * st] = fx_split(od.get());
    }
    if (C::ODD) {
      FxAcc<FXE_SHG> c;
#pragma unroll
      for (int m = 0; m < H; ++m) c.mac(a[n - 1 - m], E.mid[m]);
      g[H * st] = fx_split(c.get());
    }
  }
}

// The material products of node j's derivatives: out = r dt L (k: the level's 12 coefficients).
template <int N>
__device__ __forceinline__ void fxe_node(const fx2* G, const fx2* kc, int j, long long (&out)[9],
                                         unsigned& big) {
  constexpr int NSP = CfgE<N>::NSP;
  const auto g = [&](int d, int i) { return G[(d * 6 + i) * NSP + j]; };
  const auto k = [&](int i) {
    const fx2 c = kc[i];
    return fx3{c.h, c.l, c.l >> 16};
  };
#pragma unroll
  for (int i = 0; i < 3; ++i) {  // velocities: sum_d d sigma_{id} / dx_d
    FxAcc<FXE_SHC> a;
#pragma unroll
    for (int d = 0; d < 3; ++d) a.mac(g(d, 3 + i), k(d * 4));
    out[i] = a.get();
  }
  {
    const fx2 e[3] = {g(0, 0), g(1, 1), g(2, 2)};
#pragma unroll
    for (int i = 0; i < 3; ++i) {  // normal stresses
      FxAcc<FXE_SHC> a;
#pragma unroll
      for (int d = 0; d < 3; ++d) a.mac(e[d], k(d * 4 + (i == d ? 1 : 2)));
      out[3 + i] = a.get();
    }
  }
#pragma unroll
  for (int v = 6; v < 9; ++v) {  // shear stress of the directions (da, db)
    const int da = v == 8 ? 1 : 0, db = v == 6 ? 1 : 2;
    FxAcc<FXE_SHC> a;
    a.mac(g(da, db), k(da * 4 + 3));
    a.mac(g(db, da), k(db * 4 + 3));
    out[v] = a.get();
  }
#pragma unroll
  for (int v = 0; v < 9; ++v) {
    const int h = (int)(out[v] >> 32);
    big |= (unsigned)(h ^ (h >> 31));
  }
}

// Binary32 derivatives of every line; LO: with the table's lo parts.
template <int N, bool LO>
__device__ __forceinline__ void fxe_lines_f(const TablesE& E, const float* X, float* G, const FxeLines<N>& L) {
  using C = CfgE<N>;
  constexpr int n = C::n, H = C::H;
#pragma unroll
  for (int r = 0; r < FxeLines<N>::RND; ++r) {
    int px, pg, st;
    if (!L.get(r, px, pg, st)) continue;
    const float* x = X + px;
    float* g = G + pg;
    float a[n];
#pragma unroll
    for (int m = 0; m < n; ++m) a[m] = x[m * st];
    const auto mac = [](float& h, float& l, float2 t, float y) {
      h = fmaf(t.x, y, h);
      if (LO) l = fmaf(t.y, y, l);
    };
#pragma unroll
    for (int k = 0; k < H; ++k) {
      float ev = 0.f, od = 0.f, el = 0.f, ol = 0.f;
#pragma unroll
      for (int m = 0; m < H; ++m) {
        mac(ev, el, E.evf[k][m], a[n - 1 - m]);
        mac(od, ol, E.odf[k][m], a[m]);
      }
      if (C::ODD) mac(od, ol, E.odf[k][H], a[H]);
      g[k * st] = LO ? ev + el : ev;
      g[(n - 1 - k) * st] = LO ? od + ol : od;
    }
    if (C::ODD) {
      float c = 0.f, cl = 0.f;
#pragma unroll
      for (int m = 0; m < H; ++m) mac(c, cl, E.midf[m], a[n - 1 - m]);
      g[H * st] = LO ? c + cl : c;
    }
  }
}

// The material products in binary32 (k: dt times the coefficients as (hi, lo) pairs, r: the level's
// factor).
template <int N, bool LO>
__device__ __forceinline__ void fxe_node_f(const float* G, const float2* k, float r, int j,
                                           float (&out)[9]) {
  constexpr int NSP = CfgE<N>::NSP;
  const auto mac = [&](float& o, int c, float g) {
    o = LO ? fmaf(k[c].x, g, fmaf(k[c].y, g, o)) : fmaf(k[c].x, g, o);
  };
  const auto g = [&](int d, int i) { return G[(d * 6 + i) * NSP + j]; };
#pragma unroll
  for (int i = 0; i < 9; ++i) out[i] = 0.f;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
#pragma unroll
    for (int i = 0; i < 3; ++i) mac(out[i], d * 4, g(d, 3 + i));
    const float e = g(d, d);
#pragma unroll
    for (int i = 0; i < 3; ++i) mac(out[3 + i], d * 4 + (i == d ? 1 : 2), e);
#pragma unroll
    for (int v = 6; v < 9; ++v) {
      const int s = Elastic::src(d, v);
      if (s >= 0) mac(out[v], d * 4 + 3, g(d, s));
    }
  }
#pragma unroll
  for (int i = 0; i < 9; ++i) out[i] *= r;
}

// The CPB cells from c0 (one block); false (for every thread) when the block needs the other form.
// MIXED: the levels after the first, of the size of the step squared and less, in binary32.
template <int N, bool MIXED>
__device__ __forceinline__ bool predictor_elastic_fx(const StepArgs& A, const TablesE& E,
                                                     long long c0) {
  using C = CfgE<N>;
  constexpr int n = C::n, NS = C::NS, NV = C::NV, NL = C::NL, NF = C::NF, CPB = C::CPB;
  constexpr int NSP = C::NSP, M = C::M, H = C::H, FR = NF * NV;
  extern __shared__ __align__(16) double smem[];
  const int ncb = (int)(A.g.ncells - c0 < CPB ? A.g.ncells - c0 : CPB);
  const long long sc = A.src.cell - c0;
  if (A.nfx <= 0 || (sc >= 0 && sc < ncb)) return false;
  __shared__ int s_e[CPB];
  __shared__ float2 s_kf[MIXED ? CPB : 1][12];
  fx2(*s_k)[fxe_levels(N) + 1][12] =  // the levels' coefficients
      reinterpret_cast<fx2(*)[fxe_levels(N) + 1][12]>(reinterpret_cast<unsigned char*>(smem) + CPB * C::CELL);
  const int tid = threadIdx.x;
  const int slot = tid / NS, j = tid - slot * NS;
  const bool act = slot < ncb;
  const long long c = c0 + slot;
  fx2* X = reinterpret_cast<fx2*>(smem) + (size_t)(act ? slot : 0) * (C::CELL / sizeof(fx2));  // [9][NSP]
  fx2* G = X + 9 * NSP;                                                          // [18][NSP]
  double* stage = reinterpret_cast<double*>(G);
  const int K = A.nfx;
  const double dt = A.dev->dt;
  const double* u = A.u + c * NL;
  if (tid < CPB) s_e[tid] = 200;
  int over = 0, ez = 0;
  unsigned big = 0;
  __syncthreads();
  if (act) {
    const double rho = A.mat[c * 3], lam = A.mat[c * 3 + 1], mu = A.mat[c * 3 + 2];
    // 2^ez: the power of two below the impedance rho vp
    const float z = sqrtf(__double2float_rn(rho) * __double2float_rn(lam + 2.0 * mu));
    const unsigned zb = __float_as_uint(z);
    if (!(zb > 0x0d800000u && zb < 0x71800000u)) over = -1;  // 2^-100 .. 2^100
    ez = (int)((zb >> 23) & 255u) - 127;
    const double s = __hiloint2double((1023 + ez) << 20, 0), is = __hiloint2double((1023 - ez) << 20, 0);
    for (int i = j; i < 12 * (K + 1); i += NS) {
      const int k = i / 12, q = i % 4, d = (i % 12) / 4;
      const double m = q == 0 ? s / rho : is * (q == 1 ? lam + 2.0 * mu : (q == 2 ? lam : mu));
      s_k[slot][k][i % 12] = fx_split(fx_in(dt * A.rfx[k] * A.g.inv_h[d] * m, 1082 - E.kc, over));
      if (MIXED && k == K) {
        const ff x = ff_split(dt * A.g.inv_h[d] * m);
        s_kf[slot][i % 12] = make_float2(x.h, x.l);
      }
    }
    // the cell's state, coalesced, and its largest exponent (stresses over 2^ez)
    int emax = 200;
    for (int r = j; r < NL; r += NS) {
      const double x = u[r];
      stage[r] = x;
      const int e = (int)(((unsigned)__double2hiint(x) >> 20) & 0x7ffu);
      if (e == 0x7ff) over = -1;
      const int es = e - (r % NV >= 3 ? ez : 0);
      emax = es > emax ? es : emax;
    }
    atomicMax(&s_e[slot], emax);
  }
  __syncthreads();
  const int Ec = s_e[act ? slot : 0];
  if (Ec > 1900) over = -1;  // results near an end of binary64's range
  // (the mixed form's node form loses values below 2^-126, as its float-float pairs do)
  if (!MIXED && act && Ec < 300) over |= fxe_tiny(stage, j, NL, NS);
  // octets of mirrored nodes: into fixed point and the parity basis
  if (act) {
    for (int g = j; g < NV * M * M * M; g += NS) {
      const int v = g % NV, o = g / NV;
      const int a = o % M, b = (o / M) % M, w = o / (M * M);
      const int Ev = Ec + (v >= 3 ? ez : 0);
      long long x[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int ja = i & 1 ? n - 1 - a : a, jb = i & 2 ? n - 1 - b : b, jw = i & 4 ? n - 1 - w : w;
        x[i] = fx_in<4>(stage[(ja + n * (jb + n * jw)) * NV + v], Ev, over);
      }
      fx_octet(x);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int ja = i & 1 ? n - 1 - a : a, jb = i & 2 ? n - 1 - b : b, jw = i & 4 ? n - 1 - w : w;
        // a middle node is its own mirror: the sum (twice the value) stays, the difference goes
        if (C::ODD && (((i & 1) && a == H) || ((i & 2) && b == H) || ((i & 4) && w == H))) continue;
        X[v * NSP + ja + n * (jb + n * jw)] = fx_split(x[i]);
      }
    }
  }
  __syncthreads();
  long long S[NV];  // qbar: the sum of the levels at this node (parity index)
#pragma unroll
  for (int v = 0; v < NV; ++v) S[v] = act ? fx_join(X[v * NSP + j]) : 0;
  const FxeLines<N> L(j);
  const int KI = MIXED ? 1 : K;  // levels in fixed point
  float d32[MIXED ? NV : 1];     // the sum of the others
#pragma unroll 1
  for (int k = 0; k < KI; ++k) {
    if (act) fxe_lines<N>(E, X, G, L);
    __syncthreads();
    if (act) {
      long long b[NV];
      fxe_node<N>(G, s_k[slot][k], j, b, big);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        S[v] += b[v];
        if constexpr (MIXED) {
          d32[v] = 0.f;
          if (K > 1) reinterpret_cast<float*>(X)[v * NSP + j] = fx_float(b[v]);
          else X[v * NSP + j] = fx_split(S[v]);
        } else {
          X[v * NSP + j] = fx_split(k == K - 1 ? S[v] : b[v]);
        }
      }
    }
    __syncthreads();
  }
  if constexpr (MIXED) {
    float* Xf = reinterpret_cast<float*>(X);
    float* Gf = reinterpret_cast<float*>(G);
#pragma unroll 1
    for (int k = 1; k < K; ++k) {
      if (act) {
        if (k == 1) fxe_lines_f<N, true>(E, Xf, Gf, L);
        else fxe_lines_f<N, false>(E, Xf, Gf, L);
      }
      __syncthreads();
      if (act) {
        float b[NV];
        if (k == 1) fxe_node_f<N, true>(Gf, s_kf[slot], (float)A.rfx[k], j, b);
        else fxe_node_f<N, false>(Gf, s_kf[slot], (float)A.rfx[k], j, b);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          d32[v] += b[v];
          if (k < K - 1) {
            Xf[v * NSP + j] = b[v];
          } else {
            // (a sum outside the scale saturates and is caught with qbar)
            S[v] += fx_from_float(fminf(fmaxf(d32[v], -0x1p61f), 0x1p61f));
            X[v * NSP + j] = fx_split(S[v]);
          }
        }
      }
      __syncthreads();
    }
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const int h = (int)(S[v] >> 32);
    big |= (unsigned)(h ^ (h >> 31));
  }
  // dt L qbar
  long long* W = reinterpret_cast<long long*>(G);  // [9][NSP]
  if (act) fxe_lines<N>(E, X, G, L);
  __syncthreads();
  {
    long long b[NV];
    if (act) fxe_node<N>(G, s_k[slot][K], j, b, big);
    __syncthreads();  // every node has read the derivatives
    if (act) {
#pragma unroll
      for (int v = 0; v < NV; ++v) W[v * NSP + j] = b[v];
    }
  }
  if (__syncthreads_or(over < 0 || big >= 0x10000000u)) return false;  // 2^60
  // back to the nodes (times 8): qbar in fixed point, dt L qbar as doubles
  if (act) {
    for (int g = j; g < NV * M * M * M; g += NS) {
      const int v = g % NV, o = g / NV;
      const int a = o % M, b = (o / M) % M, w = o / (M * M);
      long long x[8], y[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int ja = i & 1 ? n - 1 - a : a, jb = i & 2 ? n - 1 - b : b, jw = i & 4 ? n - 1 - w : w;
        const bool gone = C::ODD && (((i & 1) && a == H) || ((i & 2) && b == H) || ((i & 4) && w == H));
        const int p = v * NSP + ja + n * (jb + n * jw);
        x[i] = gone ? 0 : fx_join(X[p]);
        y[i] = gone ? 0 : W[p];
      }
      fx_octet(x);
      fx_octet(y);
      const int kv = Ec + (v >= 3 ? ez : 0) - 1082;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int ja = i & 1 ? n - 1 - a : a, jb = i & 2 ? n - 1 - b : b, jw = i & 4 ? n - 1 - w : w;
        if (C::ODD && (((i & 1) && a == H) || ((i & 2) && b == H) || ((i & 4) && w == H))) continue;
        const int p = v * NSP + ja + n * (jb + n * jw);
        const int h = (int)(x[i] >> 32);
        big |= (unsigned)(h ^ (h >> 31));
        X[p] = fx_split(x[i]);
        reinterpret_cast<double*>(W)[p] = fx_out(y[i], kv);
      }
    }
  }
  if (__syncthreads_or(big >= 0x20000000u)) return false;  // 2^61: room of the face values
  if (act) {
    double* un = A.u_next + c * NL;
    for (int r = j; r < NL; r += NS) {
      const int v = r % NV, p = r / NV;
      un[r] = u[r] + reinterpret_cast<const double*>(W)[v * NSP + p];
    }
    // face records: qbar extrapolated to both ends of every direction
    double* fc = A.face + c * (3 * 2 * FR);
    for (int id = j; id < 3 * FR; id += NS) {
      const int d = id / FR, r = id - d * FR;
      const int v = r % NV, jp = r / NV;
      const int st = d == 0 ? 1 : (d == 1 ? n : n * n);
      const int j0 = d == 0 ? jp * n : (d == 1 ? jp % n + (jp / n) * n * n : jp);
      const fx2* x = X + v * NSP + j0;
      FxAcc<4> f0, f1;
#pragma unroll
      for (int m = 0; m < n; ++m) {
        const fx2 a = x[m * st];
        f0.mac(a, E.e[0][m]);
        f1.mac(a, E.e[1][m]);
      }
      const int kf = Ec + (v >= 3 ? ez : 0) + E.ke;
      fc[(d * 2 + 0) * FR + r] = fx_out(f0.get(), kf);
      fc[(d * 2 + 1) * FR + r] = fx_out(f1.get(), kf);
    }
  }
  return true;
}

// The FP64 form (not inlined: its registers do not add to the integer form's).
template <int N, bool PIC>
__device__ __noinline__ void predictor_ck_plain(const StepArgs& A, const Tables& T, long long c0) {
  __syncthreads();
  predictor_ck_block<N, PIC>(A, T, c0);
}

template <int N, bool PIC>
__device__ __forceinline__ void predictor_elastic_block(const StepArgs& A, const Tables& T,
                                                        const TablesE& E, long long c0) {
  if (!predictor_elastic_fx<N, false>(A, E, c0)) predictor_ck_plain<N, PIC>(A, T, c0);
}

// The mixed predictor: u, the first level and the output in fixed point as above, the other levels in
// binary32 (of the size of the step squared and less; the second level with float-float tables).
// The node form (predictor_ck_mixed_block) keeps binary32 pairs for the first level and its FP64
// pipe time is the base term, L qbar and the face values: 54 FP64 FMAs per node of order 5 per pass.
//
// The line: Picard from order 4, Cauchy-Kowalevski from order 5.  Predictor of a step, 64^3 cells, node form -> this one, ms.  Cauchy-
// Kowalevski: order 5 16.46 -> 14.98, order 4 9.11 -> 9.09, order 3 3.88 -> 4.41, order 2 1.74 -> 2.38,
// order 1 0.42 -> 0.56; order 6 at 48^3 17.35 -> 12.45.  Picard: order 5 21.33 -> 15.51, order 4 11.03
// -> 9.36 (10^3 cells 0.0589 -> 0.0580), order 6 at 48^3 20.21 -> 12.90.  Below the conversion and the
// change of basis cost what the FMAs that they save did, or more.  Warps: 24 an SM at order 4 (28:
// 9.55, 21: 9.63), 28 above (24 and 21: 17.6 at order 5).  Error of a step against binary64: CK 5 to
// 15 times less than the node form's, Picard 1.1 to 3 times.
template <int N, bool PIC>
struct CfgEM {
  using C = CfgE<N>;
  static constexpr bool FX = N >= (PIC ? 4 : 5);
  static constexpr int TPB = C::TPB, CPB = C::CPB;
  static constexpr int MINB = FX ? (N == 4 ? 768 : 896) / TPB : CfgCKM<N>::MINB;
  static constexpr size_t SMEM =
      FX && C::SMEM_X > CfgCKM<N>::SMEM ? C::SMEM_X : CfgCKM<N>::SMEM;
  static_assert(TPB == CfgCKM<N>::TPB && CPB == CfgCKM<N>::CPB, "one launch shape for both forms");
};

// (not inlined: its registers do not add to the integer form's)
template <int N, bool PIC>
__device__ __noinline__ void predictor_ck_mixed_plain(const StepArgs& A, const Tables& T,
                                                      const TablesF& F, long long c0) {
  __syncthreads();
  predictor_ck_mixed_block<N, PIC>(A, T, F, c0);
}

template <int N, bool PIC>
__device__ __forceinline__ void predictor_elastic_mixed_block(const StepArgs& A, const Tables& T,
                                                              const TablesF& F, long long c0) {
  if constexpr (CfgEM<N, PIC>::FX) {
    if (!predictor_elastic_fx<N, true>(A, F.el, c0)) predictor_ck_mixed_plain<N, PIC>(A, T, F, c0);
  } else {
    predictor_ck_mixed_block<N, PIC>(A, T, F, c0);
  }
}

template <int N, bool PIC>
__global__ void __launch_bounds__(CfgEM<N, PIC>::TPB, CfgEM<N, PIC>::MINB)
    k_predictor_elastic_mixed(const __grid_constant__ StepArgs A, const __grid_constant__ Tables T,
                              const __grid_constant__ TablesF F) {
  predictor_elastic_mixed_block<N, PIC>(A, T, F, (long long)blockIdx.x * CfgEM<N, PIC>::CPB);
}

template <int N, bool PIC>
cudaError_t launch_predictor_elastic_mixed_n(const StepArgs& a, const Tables& t, const TablesF& f,
                                             cudaStream_t s) {
  using C = CfgEM<N, PIC>;
  static bool attr = false;
  if (!attr) {
    const cudaError_t e = cudaFuncSetAttribute(
        k_predictor_elastic_mixed<N, PIC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  const long long blocks = (a.g.ncells + C::CPB - 1) / C::CPB;
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  k_predictor_elastic_mixed<N, PIC><<<(unsigned)blocks, C::TPB, C::SMEM, s>>>(a, t, f);
  return cudaGetLastError();
}

template <int N, bool PIC>
__global__ void __launch_bounds__(CfgE<N>::TPB, CfgE<N>::MINB)
    k_predictor_elastic(const __grid_constant__ StepArgs A, const __grid_constant__ Tables T,
                        const __grid_constant__ TablesE E) {
  predictor_elastic_block<N, PIC>(A, T, E, (long long)blockIdx.x * CfgE<N>::CPB);
}

template <int N, bool PIC>
cudaError_t launch_predictor_elastic_n(const StepArgs& a, const Tables& t, const TablesF& f,
                                       cudaStream_t s) {
  using C = CfgE<N>;
  static bool attr = false;
  if (!attr) {
    const cudaError_t e = cudaFuncSetAttribute(
        k_predictor_elastic<N, PIC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  const long long blocks = (a.g.ncells + C::CPB - 1) / C::CPB;
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  k_predictor_elastic<N, PIC><<<(unsigned)blocks, C::TPB, C::SMEM, s>>>(a, t, f.el);
  return cudaGetLastError();
}

}  // namespace ader
