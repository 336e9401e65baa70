// Face-centric operator in collocation form (nq_visc = k+1: every default rule, k <= 6).
//
// The viscous Gauss points are the k+1 mass points, so the Lagrange polynomials l_g on them are an
// orthogonal basis: the mass matrix is diag(w_g |J|_g), a viscous flux at the points needs no projection,
// and every quadrature weight can be moved into the 1D tables.  With r_g the test of -F(U) against l_g
// divided by w_g, the evaluation is
//   values      U_g = S U (S the square LGL-to-Gauss matrix), U_c = S_c U at the convective points,
//   r_g      =  P (sum_d D~_d F~c_d) - sum_d D~_d F~v_d + sum over faces (l_g(0 or 1) L + l_g'(0 or 1) D) / w_g,
//               D~ = W^-1 D^T W (collocation derivative matrix D),  P[g][q] = l_g(x_q) w_q / w_g,
//   L(U)     =  S^-1 (r_g / |J|_g)  (+ the body force, pointwise before S^-1).
// Against testing with the LGL basis and then applying M^-1 = S^-1 diag(1/(|J| w)) S^-T, the three S^T
// sweeps of the viscous cell term, the three S^-T sweeps of the mass matrix and, on every face, the S^T
// sweeps of the viscous value and gradient tests cancel; the face shares (L, D) of the face buffer are
// values at the face's Gauss points.
//
// One CTA carries a batch of cells (or faces).  In FP64 the sweeps run in integer arithmetic
// (dg_fixed.cuh), so a phase that holds both sweeps and point fluxes keeps both pipes busy.  On axis-aligned
// faces the point fluxes form only the normal flux column and the nonzero entries of the jump term.
//
// Measured per launch (face / cell + stage kernel), against the kernels that test with the LGL basis and contract in
// FP64, and with the integer sweeps of both (dg_fixed.cuh):
// FP64 TGV 64^3, k = 3: 30.5 -> 24.6 -> 10.8 / 32.5 -> 21.2 -> 9.3 ms; 40^3, k = 5: 20.4 -> 14.9 -> 9.1 /
// 35.8 -> 25.7 -> 12.1 ms; FP64 channel 32^3, k = 3 (stored geometry): cell 1.65 ms (1.96 without the chains of the M^-1
// sweeps, before the share scan's loads were issued together).
// FP32 40^3, k = 5: 1.36 -> 0.88 / 2.51 -> 1.23 ms; channel 32^3, k = 3: 0.36 -> 0.24 / 0.36 -> 0.24 ms;
// FP32 64^3, k = 3, cell + stage: 2.14 (register-resident tasks, one cell per CTA) -> 1.39 ms.
// Bound by: FP64 faces the FP64 pipe in the point phases (63 % busy overall) and latency; FP64 cells latency (FP64 pipe
// 49 %, ALU 42 %, four CTAs per SM); FP32 shared-memory wavefronts (89 %) and issue (62 %).
#pragma once
#include "dg_chain.cuh"
#include "dg_faces.cuh"
#include "dg_kernels.cuh"

namespace dgcns {

// ---------------------------------------------------------------------------
// Sweeps.  nblk blocks of (D2, D1, D0) values (D0 fastest), the planes of D1 x D0 values IPS apart; the operator
// acts along axis AX, the output's planes are OPS apart.  NIN: the input is the sum of NIN arrays ks apart (and
// of `extra` when EX).  IBS > 0: blocks IBS apart in the input; OBS > 0: in the output (an in-place sweep that
// keeps its block stride).
//
// FP32 planes whose rows are 8 values (k = 5: QC = 8) are padded so that the lines along y of 32 lanes (D0 neighbours, then the
// next plane) fall on distinct banks, and lines along x are read as 16- or 8-byte vectors: with dense planes at k = 3, 43 % of the
// cell kernel's shared-memory wavefronts were conflicts and that pipe was 82 % busy.  FP64 planes are dense (the
// padding would cost a resident CTA; its kernels keep that pipe 30 % busy).
// ---------------------------------------------------------------------------
template <typename T>
constexpr int plane_stride(int d0, int d1) {
  if (sizeof(T) == 8) return d0 * d1;
  if (d0 % 8 != 0) return d0 * d1;
  int best = d0 * d1, bestc = 99;
  for (int s = d0 * d1; s <= d0 * d1 + 12; s += 4) {
    int cnt[32] = {}, c = 0;
    for (int l = 0; l < 32; ++l) {
      const int k = (l % d0 + l / d0 * s) % 32;
      if (++cnt[k] > c) c = cnt[k];
    }
    if (c < bestc) {
      bestc = c;
      best = s;
    }
  }
  return best;
}

// K consecutive values with the widest aligned vectors the extent allows (arrays start on 16 bytes).
template <typename T, int K, bool LD>
__device__ __forceinline__ void line_io(T* p, T (&x)[K]) {
  if constexpr ((K * sizeof(T)) % 16 == 0) {
    if constexpr (LD)
      vec_load<T, K>(p, x);
    else
      vec_store<T, K>(p, x);
  } else if constexpr (sizeof(T) == 4 && K % 2 == 0) {
#pragma unroll
    for (int i = 0; i < K; i += 2) {
      if constexpr (LD) {
        const float2 v = *reinterpret_cast<const float2*>(p + i);
        x[i] = v.x;
        x[i + 1] = v.y;
      } else {
        *reinterpret_cast<float2*>(p + i) = make_float2(x[i], x[i + 1]);
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < K; ++i) {
      if constexpr (LD)
        x[i] = p[i];
      else
        p[i] = x[i];
    }
  }
}

// FP64 line by line (what a chain cannot take, and stored geometry's last sweeps): line l = (outer, inner) with
// inner < n0 starts at outer n0 DIN + inner.  One function per shape, not inlined (the code of an integer line is
// long; the axes share it).  OG: OG consecutive outers form a block, blocks IBS apart.
template <int DIN, int DOUT, int SYM, int NIN, bool EX, int OG, int IBS, int OBS>
__device__ __noinline__ void lines_fp64(const double* in, int ks, const double* extra, double* out, EoFp64 E, int nlines,
                                        int n0, uint32_t magic) {
  DGCNS_SHARED(in);
  DGCNS_SHARED(out);
  DGCNS_SHARED(E.f);
  DGCNS_SHARED(E.p);
#pragma unroll 1
  for (int l = threadIdx.x; l < nlines; l += blockDim.x) {
    const int outer = n0 > 1 ? (int)__umulhi((uint32_t)l, magic) : l;
    const int inner = l - outer * n0;
    const int ib = (OG > 0 ? (outer / (OG > 0 ? OG : 1)) * IBS + (outer % (OG > 0 ? OG : 1)) * n0 * DIN : outer * n0 * DIN) + inner;
    const int ob = (OBS > 0 ? outer * OBS : outer * n0 * DOUT) + inner;
    constexpr int NA = NIN + (EX ? 1 : 0);
    double x[NA][DIN], y[DOUT];
#pragma unroll
    for (int a = 0; a < NA; ++a) {
      const double* p = EX && a == NIN ? extra + ib : in + ib + (size_t)a * ks;
#pragma unroll
      for (int i = 0; i < DIN; ++i) x[a][i] = p[i * n0];
    }
    line_apply_sum<double, NA, DIN, DOUT, SYM>(E, x, y);
#pragma unroll
    for (int q = 0; q < DOUT; ++q) out[ob + q * n0] = y[q];
  }
}

template <typename T, int AX, int D0, int D1, int D2, int DOUT, int SYM, int IPS = D0 * D1,
          int OPS = (AX == 0 ? DOUT * D1 : (AX == 1 ? D0 * DOUT : D0 * D1)), int NIN = 1, bool EX = false, int IBS = 0,
          int OBS = 0>
__device__ __forceinline__ void sw(const T* in, T* out, Eo<T> E, int nblk, int ks = 0, const T* extra = nullptr) {
  constexpr int DIN = AX == 0 ? D0 : (AX == 1 ? D1 : D2);
  constexpr int n0 = AX == 0 ? 1 : (AX == 1 ? D0 : D0 * D1);  // values below the axis
  constexpr int per = AX == 0 ? D1 * D2 : (AX == 1 ? D2 : 1);  // groups of n0 lines per block
  if constexpr (sizeof(T) == 8) {
    constexpr uint32_t magic = n0 > 1 ? (uint32_t)((0x100000000ull + n0 - 1) / n0) : 0u;  // l / n0 for l n0 < 2^32
    lines_fp64<DIN, DOUT, SYM, NIN, EX, (IBS > 0 ? per : 0), IBS, OBS>(in, ks, extra, out, E, nblk * per * n0, n0, magic);
  } else {
    constexpr int NA = NIN + (EX ? 1 : 0);
    constexpr int ist = AX == 0 ? 1 : (AX == 1 ? D0 : IPS), ost = AX == 0 ? 1 : (AX == 1 ? D0 : OPS);
    // lines along x: row l of plane l / D1; along y: neighbour `inner` of plane g; along z: of block g
    constexpr int igs = AX == 1 ? IPS : D2 * IPS, ogs = AX == 1 ? OPS : (OBS > 0 ? OBS : DOUT * OPS);
    for (int l = threadIdx.x; l < nblk * per * n0; l += blockDim.x) {
      const int g = l / n0, inner = l - g * n0;
      int ib, ob;
      if constexpr (AX == 0) {
        ib = l * D0 + l / D1 * (IPS - D0 * D1);
        ob = l * DOUT + l / D1 * (OPS - DOUT * D1);
      } else {
        ib = (IBS > 0 ? g / per * IBS + g % per * IPS : g * igs) + inner;
        ob = g * ogs + inner;
      }
      T x[NA][DIN], y[DOUT];
#pragma unroll
      for (int a = 0; a < NA; ++a) {
        const T* p = EX && a == NIN ? extra + ib : in + ib + (size_t)a * ks;
        if constexpr (AX == 0) {
          line_io<T, DIN, true>(const_cast<T*>(p), x[a]);
        } else {
#pragma unroll
          for (int i = 0; i < DIN; ++i) x[a][i] = p[i * ist];
        }
      }
      line_apply_sum<T, NA, DIN, DOUT, SYM>(E, x, y);
      if constexpr (AX == 0) {
        line_io<T, DOUT, false>(out + ob, y);
      } else {
#pragma unroll
        for (int q = 0; q < DOUT; ++q) out[ob + q * ost] = y[q];
      }
    }
  }
}

// V_d <- D~_d V_d + the shares of the two faces of direction d, in place.  V: [nb][5][N][N, N]; F: the cells' face
// shares [nb][6][2][5][N^2] (global).  The line's operator takes D_0, L_0, the N values, -L_1, D_1: with the sign
// of L_1 it is antisymmetric under reflection like D~ itself.
template <typename T, int N, int D>
__device__ __forceinline__ void lift_body(T* V, const T* F, Eo<T> E, int nb, bool vol) {
  constexpr int N2 = N * N, PS = plane_stride<T>(N, N), st = D == 0 ? 1 : (D == 1 ? N : PS);
  for (int l = threadIdx.x; l < nb * 5 * N2; l += blockDim.x) {
    const int ec = l / N2, j = l - ec * N2, e = ec / 5, c = ec - 5 * e, j1 = j % N, j2 = j / N;
    const T* f0 = F + (size_t)e * fbuf_per_cell<N>() + (2 * D * 2 * 5 + c) * N2 + j;
    const T* f1 = f0 + 2 * 5 * N2;
    T x[N + 4], y[N];
    x[0] = f0[5 * N2];
    x[1] = f0[0];
    x[N + 2] = -f1[0];
    x[N + 3] = f1[5 * N2];
    T* v = V + ec * N * PS + (D == 0 ? j1 * N + j2 * PS : (D == 1 ? j1 + j2 * PS : j1 + N * j2));
    if constexpr (D == 0) {
      line_io<T, N, true>(v, y);
    } else {
#pragma unroll
      for (int i = 0; i < N; ++i) y[i] = v[i * st];
    }
#pragma unroll
    for (int i = 0; i < N; ++i) x[2 + i] = vol ? y[i] : T(0);
    line_apply<T, N + 4, N, -1>(E, x, y);
    if constexpr (D == 0) {
      line_io<T, N, false>(v, y);
    } else {
#pragma unroll
      for (int i = 0; i < N; ++i) v[i * st] = y[i];
    }
  }
}
template <int N>
__device__ __noinline__ void lift_fp64(double* V, const double* F, EoFp64 E, int nb, bool vol, int n3) {
  DGCNS_SHARED(V);
  DGCNS_SHARED(E.f);
  DGCNS_SHARED(E.p);
  // the three directions one after the other, V_d n3 values apart
  lift_body<double, N, 0>(V, F, E, nb, vol);
  lift_body<double, N, 1>(V + n3, F, E, nb, vol);
  lift_body<double, N, 2>(V + 2 * n3, F, E, nb, vol);
}

// ---------------------------------------------------------------------------
// Point fluxes
// ---------------------------------------------------------------------------
// Convective flux w F_c . n of one side of a face and its wave speed (LLF); n any unit normal, or e_D when AFF (w then
// carries the sign).  Components in physical order.
template <typename T, int D, bool AFF>
__device__ __forceinline__ void llf_side(const T u[5], const T n[3], T w, const PhysT<T>& ph, T f[5], T& lam) {
  const T rinv = rcp_of(ph.rho_r + u[0]);
  const T m2 = u[1] * u[1] + u[2] * u[2] + u[3] * u[3];
  const T dp = ph.gm1 * u[4] - (ph.hgm1 * rinv) * m2;
  lam = sqrt_of(m2) * rinv + sqrt_of(fabs((ph.g_pr + ph.gamma * dp) * rinv));
  const T mn = w * (AFF ? u[1 + D] : u[1] * n[0] + u[2] * n[1] + u[3] * n[2]);
  const T vn = mn * rinv;
  f[0] = mn;
  f[1] = u[1] * vn;
  f[2] = u[2] * vn;
  f[3] = u[3] * vn;
  if (AFF) {
    f[1 + D] += w * dp;
  } else {
    const T wp = w * dp;
    f[1] += wp * n[0];
    f[2] += wp * n[1];
    f[3] += wp * n[2];
  }
  f[4] = (ph.H_r + u[4] + dp) * vn;
}

// Velocity, energy and reciprocal density of one side.
template <typename T>
struct SideState {
  T rinv, v[3], E;
};
template <typename T>
__device__ __forceinline__ SideState<T> side_state(const T u[5], const PhysT<T>& ph) {
  SideState<T> s;
  s.rinv = rcp_of(ph.rho_r + u[0]);
#pragma unroll
  for (int i = 0; i < 3; ++i) s.v[i] = u[1 + i] * s.rinv;
  s.E = (ph.rhoE_r + u[4]) * s.rinv;
  return s;
}

// Normal viscous flux F_v(U, G) e_D on an axis-aligned face: only the normal derivatives and, of the
// tangential ones, those of rho, m_D and the tangential momentum along its own direction enter.  All derivatives are
// reference ones (times hinv).  gd: along the normal (physical order); r1, d1, a1: along t1 of rho, m_D, m_t1; r2, d2,
// a2: along t2 of rho, m_D, m_t2.  f: components (m_D, m_t1, m_t2, rho E).
template <typename T, int D>
__device__ __forceinline__ void visc_normal(const SideState<T>& s, const T gd[5], T r1, T d1, T a1, T r2, T d2, T a2,
                                            const KConst<T>& kc, T f[4]) {
  constexpr int t1 = D == 0 ? 1 : 0, t2 = D == 2 ? 1 : 2;
  const T rd = kc.hinv[D] * s.rinv, ra = kc.hinv[t1] * s.rinv, rb = kc.hinv[t2] * s.rinv;
  const T ad = (gd[1 + D] - s.v[D] * gd[0]) * rd;
  const T at1 = (gd[1 + t1] - s.v[t1] * gd[0]) * rd;
  const T at2 = (gd[1 + t2] - s.v[t2] * gd[0]) * rd;
  const T cc = (a1 - s.v[t1] * r1) * ra + (a2 - s.v[t2] * r2) * rb;
  f[0] = kc.mu43 * ad - kc.mu23 * cc;
  f[1] = kc.mu * (at1 + (d1 - s.v[D] * r1) * ra);
  f[2] = kc.mu * (at2 + (d2 - s.v[D] * r2) * rb);
  const T q = (gd[4] - s.E * gd[0]) * rd - (s.v[D] * ad + s.v[t1] * at1 + s.v[t2] * at2);
  f[3] = f[0] * s.v[D] + f[1] * s.v[t1] + f[2] * s.v[t2] + kc.lam_cv * q;
}

// Integrands of +1/2 (grad V, F_v(U, j (x) e_D)) on an axis-aligned face over the cell's |J|: normal column
// fd (m_D, m_t1, m_t2, rho E) and the nonzero entries (m_D, m_t, rho E) of the tangential columns, with all
// constant factors (mu/2, 1/h of both directions) in kc.mus and kc.lams.
template <typename T, int D>
__device__ __forceinline__ void visc_jump(const SideState<T>& s, const T j[5], const KConst<T>& kc, T fd[4], T f1[3],
                                          T f2[3]) {
  constexpr int t1 = D == 0 ? 1 : 0, t2 = D == 2 ? 1 : 2;
  const T gd = j[1 + D] - s.v[D] * j[0];
  const T g1 = j[1 + t1] - s.v[t1] * j[0];
  const T g2 = j[1 + t2] - s.v[t2] * j[0];
  const T rd = kc.mus[D][D] * s.rinv, ra = kc.mus[D][t1] * s.rinv, rb = kc.mus[D][t2] * s.rinv;
  fd[0] = (kc.mus43[D] * s.rinv) * gd;
  fd[1] = rd * g1;
  fd[2] = rd * g2;
  const T vg = s.v[D] * gd + s.v[t1] * g1 + s.v[t2] * g2;
  fd[3] = fd[0] * s.v[D] + fd[1] * s.v[t1] + fd[2] * s.v[t2] + (kc.lams[D] * s.rinv) * (j[4] - s.E * j[0] - vg);
  f1[0] = ra * g1;
  f1[1] = -(kc.mus23[D][t1] * s.rinv) * gd;
  f1[2] = f1[0] * s.v[D] + f1[1] * s.v[t1];
  f2[0] = rb * g2;
  f2[1] = -(kc.mus23[D][t2] * s.rinv) * gd;
  f2[2] = f2[0] * s.v[D] + f2[1] * s.v[t2];
}

// F_v(U, G) n for a general unit normal; rows of f: momenta and energy.
template <typename T>
__device__ __forceinline__ void visc_normal_any(const SideState<T>& s, const T G[5][3], const T n[3],
                                                const PhysT<T>& ph, T f[4]) {
  T gn[5];
#pragma unroll
  for (int c = 0; c < 5; ++c) gn[c] = G[c][0] * n[0] + G[c][1] * n[1] + G[c][2] * n[2];
  const T vn = s.v[0] * n[0] + s.v[1] * n[1] + s.v[2] * n[2];
  T a[3], b[3], div = T(0);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    a[i] = (gn[1 + i] - s.v[i] * gn[0]) * s.rinv;  // (grad u) n
    b[i] = (n[0] * G[1][i] + n[1] * G[2][i] + n[2] * G[3][i] - vn * G[0][i]) * s.rinv;  // (grad u)^T n
    div += G[1 + i][i] - s.v[i] * G[0][i];
  }
  div *= T(2) / T(3) * s.rinv;
#pragma unroll
  for (int i = 0; i < 3; ++i) f[i] = ph.mu * (a[i] + b[i] - div * n[i]);
  const T q = (gn[4] - s.E * gn[0]) * s.rinv - (s.v[0] * a[0] + s.v[1] * a[1] + s.v[2] * a[2]);
  f[3] = f[0] * s.v[0] + f[1] * s.v[1] + f[2] * s.v[2] + ph.lam_cv * q;
}

// F_v(U, j (x) n) contracted with a row J of the inverse Jacobian: tau = mu (g (x) n + n (x) g - 2/3 (g.n) I),
// g = (j_m - v j_0)/rho.  Per side: g, g.n, the energy coefficient; per row three momenta and the energy.
template <typename T>
struct JumpFlux {
  T g[3], h, q;
};
template <typename T>
__device__ __forceinline__ JumpFlux<T> visc_jump_any(const SideState<T>& s, const T j[5], const T n[3],
                                                     const PhysT<T>& ph) {
  JumpFlux<T> r;
  const T mr = ph.mu * s.rinv;
  T vg = T(0);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const T g = j[1 + i] - s.v[i] * j[0];
    vg += s.v[i] * g;
    r.g[i] = mr * g;
  }
  r.h = T(-2) / T(3) * (r.g[0] * n[0] + r.g[1] * n[1] + r.g[2] * n[2]);
  r.q = (ph.lam_cv * s.rinv) * (j[4] - s.E * j[0] - vg);
  return r;
}
template <typename T>
__device__ __forceinline__ void jump_row(const JumpFlux<T>& r, const SideState<T>& s, const T n[3], const T* J, T w,
                                         T f[4]) {
  const T nj = n[0] * J[0] + n[1] * J[1] + n[2] * J[2];
  const T gj = r.g[0] * J[0] + r.g[1] * J[1] + r.g[2] * J[2];
#pragma unroll
  for (int i = 0; i < 3; ++i) f[i] = r.g[i] * nj + n[i] * gj + r.h * J[i];
  f[3] = w * (f[0] * s.v[0] + f[1] * s.v[1] + f[2] * s.v[2] + r.q * nj);
#pragma unroll
  for (int i = 0; i < 3; ++i) f[i] *= w;
}

// ---------------------------------------------------------------------------
// Cell kernel
// ---------------------------------------------------------------------------
// Shared memory per cell: the three convective flux arrays [3][5][QC^3] (their space also holds the nodal
// state, the interpolation temporaries, the projected residual and M^-1's temporaries) and the viscous
// point arrays [3][5][N^3] (gradients, then fluxes) with the values U_g [5][N^3].
template <typename T, int N, int QC>
struct CollSizes {
  static constexpr int N2 = N * N, N3 = N2 * N, PC = QC * QC * QC;
  // plane strides of the point and node arrays, and of the (QC x, N y) planes; block sizes
  static constexpr int PN = plane_stride<T>(N, N), PQ = plane_stride<T>(QC, QC), P1 = plane_stride<T>(QC, N);
  static constexpr int BN = N * PN, BQ = QC * PQ;
  static constexpr int F0 = BQ > BN ? BQ : BN, F1 = N * P1 > F0 ? N * P1 : F0;
  static constexpr int F = (F1 + 3) & ~3;
  static constexpr int PER_CELL = 15 * F + 20 * BN;
};
template <typename T, int N, int QC, int QV, int CB>
constexpr size_t coll_cell_smem() {
  return ((size_t)table_elems<T, N, QC, QV>() + (size_t)CB * CollSizes<T, N, QC>::PER_CELL) * sizeof(T) +
         (sizeof(T) == 8 ? 25 * CB * sizeof(uint32_t) : 0) + 64;
}

// Cells per CTA and threads.
template <typename T, int N, int QC, int QV>
constexpr int coll_cells() {
  int cb = 2;
  while (cb > 1 && ((size_t)table_elems<T, N, QC, QV>() + (size_t)cb * CollSizes<T, N, QC>::PER_CELL) * sizeof(T) > 74 * 1024)
    --cb;
  return cb;
}
// Threads: 128, and more where only two (FP64) or four (FP32) large cells fit an SM.  Measured: FP64 k = 3, 2 cells
// and 128 threads 14.9 ms per stage at 64^3 (192 threads 17.4, one cell 17.9 to 23.6), before the chains, now 9.3;
// FP64 k = 5, 40^3, 192 threads 15.2 ms (128: 18.5, 256: 27.0, their registers no longer hold the point fluxes), now
// 12.1; FP32 k = 5, 256 threads 1.30 ms (128: 1.67, 192: 1.34), now 1.23; FP32 k = 3 stored, 32^3, 2 cells and 128
// threads 0.264 ms (256: 0.326; one cell 0.277).
template <typename T, int N, int QC, int QV>
constexpr int coll_threads() {
  constexpr size_t smem = coll_cell_smem<T, N, QC, QV, coll_cells<T, N, QC, QV>()>();
  return sizeof(T) == 8 ? (smem > 64 * 1024 ? 192 : 128) : (smem > 40 * 1024 ? 256 : 128);
}
template <typename T, int N, int QC, int QV, int CB>
constexpr int coll_ctas() {  // resident CTAs that the registers have to allow
  const int b = (int)(227 * 1024 / coll_cell_smem<T, N, QC, QV, CB>());
  return b < 1 ? 1 : (b > 4 ? 4 : b);
}

// kp.out_mode: 0 writes F(U), 1 L(U), 2 the stage update (as dg_op_kernel).
template <typename T, int N, int QC, int QV, int CB, int GEO>
__global__ void __launch_bounds__(coll_threads<T, N, QC, QV>(), coll_ctas<T, N, QC, QV, CB>())
    dg_coll_cell_kernel(const KParams kp, const double* U,
                                                                         T* Rout, T* dU, double* Uout) {
  static_assert(QV == N && GEO != GEO_FLY, "collocation form");
  using S = CollSizes<T, N, QC>;
  constexpr int N2 = S::N2, N3 = S::N3, PC = S::PC, PN = S::PN, PQ = S::PQ, P1 = S::P1, BN = S::BN, BQ = S::BQ;
  constexpr int QC2 = QC * QC, NTH = coll_threads<T, N, QC, QV>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* stab = reinterpret_cast<T*>(smem_raw);
  T* F0 = stab + table_elems<T, N, QC, QV>();
  T* F1 = F0 + CB * 5 * S::F;
  T* F2 = F1 + CB * 5 * S::F;
  T* V = F2 + CB * 5 * S::F;  // [3][CB][5][N][PN]
  constexpr int VS = CB * 5 * BN;
  T* Ug = V + 3 * VS;
  auto pad = [](int i) { return i / N2 * PN + i % N2; };  // value i of node arrays
  const int e0 = blockIdx.x * CB;
  const int nb = min(CB, kp.Nc - e0);
  const Tab<T> tb = load_tables<T, N, QC, QV>(static_cast<const T*>(kp.tables), stab);
  const PhysT<T> ph = make_phys<T>(kp);
  const KConst<T>& kc = kconst<T>(kp);
  wait_for_predecessor();
  const size_t base = (size_t)e0 * 5 * N3;
  const int nvals = nb * 5 * N3, nbl = nb * 5;
  constexpr int PER = (CB * 5 * N3 + NTH - 1) / NTH;
  constexpr bool FX = sizeof(T) == 8;  // integer chains
  const T* Ud = static_cast<const T*>(kp.Udev);
  const T* FBc = static_cast<const T*>(kp.fbuf) + (size_t)e0 * fbuf_per_cell<N>();
  const bool conv = kp.conv != 0, visc = kp.visc != 0;
  const bool force = kp.has_bf && kp.out_mode != 0;
  // FP64: maxima of the blocks (cell, component): of the state, of the convective flux, of the viscous flux and the face
  // shares, of the divergence of the convective flux, of the first S^-1 sweep's result
  uint32_t* exU = reinterpret_cast<uint32_t*>(Ug + VS);
  uint32_t *exC = exU + 5 * CB, *exV = exC + 5 * CB, *exP = exV + 5 * CB, *exR = exP + 5 * CB;
  // FP64: the point phases give each cell its own warps, so that a thread's maxima belong to one cell
  constexpr int NTE = FX ? NTH / CB : NTH;
  static_assert(!FX || NTE % 32 == 0, "whole warps per cell");
  const int pe = FX ? threadIdx.x / NTE : 0, pt = FX ? threadIdx.x % NTE : threadIdx.x;
  bool fixA = false, fixB = false, fixL = false, fixR = false;  // chains: values, convective flux, lift, residual and M^-1
  if constexpr (FX) {
    constexpr int PV = (N3 + NTE - 1) / NTE;
    const bool own = pe < nb;
    const T* sh = FBc + (own ? pe : 0) * fbuf_per_cell<N>();
    double x[5][PV];
#pragma unroll
    for (int c = 0; c < 5; ++c)
#pragma unroll
      for (int k = 0; k < PV; ++k) {
        const int i = k * NTE + pt;
        x[c][k] = own && i < N3 ? U[base + (pe * 5 + c) * N3 + i] : 0.0;
      }
    if (threadIdx.x < 25 * CB) exU[threadIdx.x] = 0;
    __syncthreads();
    uint32_t m[5], f[5];
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      m[c] = f[c] = 0;
#pragma unroll
      for (int k = 0; k < PV; ++k) {
        if ((c == 0 || c == 4) && own && k * NTE + pt < N3) x[c][k] -= c == 0 ? kp.rho_ref : kp.rhoE_ref;
        m[c] = max(m[c], fx_mag(x[c][k]));
      }
      // the shares of the batch, also brought nearer for the lift sweeps
#pragma unroll
      for (int k = 0; k < (12 * N2 + NTE - 1) / NTE; ++k) {
        // (past the end the cell's last share again, so that no load waits for a condition)
        const int i = min(k * NTE + pt, 12 * N2 - 1);
        f[c] = max(f[c], reinterpret_cast<const uint32_t*>(sh + (i / N2 * 5 + c) * N2 + i % N2)[1] & 0x7fffffffu);
      }
    }
    if (own) {
      block_max<32>(exU + pe * 5, 1, 0, m);
      block_max<32>(exV + pe * 5, 1, 0, f);
    }
    __syncthreads();
    fixA = blocks_ok(exU, 5 * CB);
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      const int E = fx_exp(exU[pe * 5 + c]);
#pragma unroll
      for (int k = 0; k < PV; ++k) {
        const int i = k * NTE + pt;
        if (own && i < N3)
          F0[(pe * 5 + c) * N3 + i] = fixA ? __longlong_as_double(fx_of(x[c][k], E)) : x[c][k];
      }
    }
  } else if (Ud) {
    batched_pass<PER>(threadIdx.x, NTH, nvals, [&](int i) { return Ud[base + i]; }, [&](int i, T v) { F0[pad(i)] = v; });
  } else {
    batched_pass<PER>(threadIdx.x, NTH, nvals, [&](int i) { return U[base + i]; }, [&](int i, double v) {
      F0[pad(i)] = dev_value<T>(kp, v, (i / N3) % 5);
    });
  }
  __syncthreads();
  // 1-3. values at the convective and at the viscous points
  int gS = 0;  // exponent of U_g over the state's (chains)
  if (FX && fixA) {
    if constexpr (FX) {
      const int gC = chain_gain(tb.eSc);
      gS = chain_gain(tb.eSm);
      if (conv) chain<1, N, QC, 1, FROM_INT, TO_INT, N2>(F0, F1, tb.eSc, nbl * N2, exU, 0);
      chain<1, N, N, 1, FROM_INT, TO_INT, N2>(F0, V, tb.eSm, nbl * N2, exU, 0);
      __syncthreads();
      if (conv) chain<QC, N, QC, 1, FROM_INT, TO_INT, QC * N>(F1, F2, tb.eSc, nbl * N, exU, 0);
      chain<N, N, N, 1, FROM_INT, TO_INT, N2>(V, V + VS, tb.eSm, nbl * N, exU, 0);
      __syncthreads();
      if (conv) chain<QC * QC, N, QC, 1, FROM_INT, TO_DOUBLE, QC2>(F2, F0, tb.eSc, nbl, exU, 2 * gC);
      chain<N2, N, N, 1, FROM_INT, TO_INT, N2>(V + VS, Ug, tb.eSm, nbl, exU, 0);
      gS *= 3;
    }
  } else {
    if (conv) sw<T, 0, N, N, N, QC, 1, PN, P1>(F0, F1, tb.eSc, nbl);
    sw<T, 0, N, N, N, N, 1, PN, PN>(F0, V, tb.eSm, nbl);
    __syncthreads();
    if (conv) sw<T, 1, QC, N, N, QC, 1, P1, PQ>(F1, F2, tb.eSc, nbl);
    sw<T, 1, N, N, N, N, 1, PN, PN>(V, V + VS, tb.eSm, nbl);
    __syncthreads();
    if (conv) sw<T, 2, QC, QC, N, QC, 1, PQ, PQ>(F2, F0, tb.eSc, nbl);
    sw<T, 2, N, N, N, N, 1, PN, PN>(V + VS, Ug, tb.eSm, nbl);
  }
  __syncthreads();
  auto ug = [&](int i, int b) -> T {  // value i of U_g, in block b
    if constexpr (FX) {
      if (fixA) return fx_store(__double_as_longlong(Ug[i]), fx_exp(exU[b]) + gS + 3);
    }
    return Ug[i];
  };
  uint32_t mag[5] = {0, 0, 0, 0, 0};
  auto see = [&](int c, T v) {
    if constexpr (FX) mag[c] = max(mag[c], fx_mag(v));
    return v;
  };
  // 4. convective flux (point arithmetic); reference gradients at the viscous points (sweeps)
  if (conv) {
    for (int idx = pt; idx < (FX ? (pe < nb ? PC : 0) : nb * PC); idx += NTE) {
      const int e = FX ? pe : idx / PC, p = FX ? idx : idx - e * PC, o = e * 5 * BQ + p / QC2 * PQ + p % QC2;
      T u[5];
#pragma unroll
      for (int c = 0; c < 5; ++c) u[c] = F0[o + c * BQ];
      const T rinv = rcp_of(ph.rho_r + u[0]);
      const T dp = ph.gm1 * u[4] - (ph.hgm1 * rinv) * (u[1] * u[1] + u[2] * u[2] + u[3] * u[3]);
      const T Hr = (ph.H_r + u[4] + dp) * rinv;
      T* Fd[3] = {F0, F1, F2};
      if (GEO == GEO_AFFINE) {
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const T m = kc.hinv[j] * u[1 + j];
          const T a = m * rinv;
          T* f = Fd[j] + o;
          f[0] = see(0, m);
#pragma unroll
          for (int i = 0; i < 3; ++i)
            f[(1 + i) * BQ] = see(1 + i, i == j ? u[1 + i] * a + kc.hinv[j] * dp : u[1 + i] * a);
          f[4 * BQ] = see(4, Hr * m);
        }
      } else {
        const T* g = static_cast<const T*>(kp.gcc) + (size_t)(e0 + e) * 10 * PC + p;
        const T dj = g[9 * PC];
        const T v[3] = {u[1] * rinv, u[2] * rinv, u[3] * rinv};
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          const T j0 = dj * g[(3 * b) * PC], j1 = dj * g[(3 * b + 1) * PC], j2 = dj * g[(3 * b + 2) * PC];
          const T m = j0 * u[1] + j1 * u[2] + j2 * u[3];
          T* f = Fd[b] + o;
          f[0] = see(0, m);
          f[BQ] = see(1, m * v[0] + dp * j0);
          f[2 * BQ] = see(2, m * v[1] + dp * j1);
          f[3 * BQ] = see(3, m * v[2] + dp * j2);
          f[4 * BQ] = see(4, Hr * m);
        }
      }
    }
  }
  if constexpr (FX) {
    if (conv) {
      if (pe < nb) block_max<32>(exC + pe * 5, 1, 0, mag);
#pragma unroll
      for (int c = 0; c < 5; ++c) mag[c] = 0;
    }
    if (visc && fixA) {
      chain<1, N, N, -1, FROM_INT, TO_DOUBLE, N2>(Ug, V, tb.eDv, nbl * N2, exU, gS);
      chain<N, N, N, -1, FROM_INT, TO_DOUBLE, N2>(Ug, V + VS, tb.eDv, nbl * N, exU, gS);
      chain<N2, N, N, -1, FROM_INT, TO_DOUBLE, N2>(Ug, V + 2 * VS, tb.eDv, nbl, exU, gS);
    }
  }
  if (visc && !fixA) {
    sw<T, 0, N, N, N, N, -1, PN, PN>(Ug, V, tb.eDv, nbl);
    sw<T, 1, N, N, N, N, -1, PN, PN>(Ug, V + VS, tb.eDv, nbl);
    sw<T, 2, N, N, N, N, -1, PN, PN>(Ug, V + 2 * VS, tb.eDv, nbl);
  }
  __syncthreads();
  // 5. viscous flux with the sign of -F (point arithmetic); D~ of the convective flux, in place (sweeps)
  if (visc) {
    for (int idx = pt; idx < (FX ? (pe < nb ? N3 : 0) : nb * N3); idx += NTE) {
      const int e = FX ? pe : idx / N3, p = FX ? idx : idx - e * N3, o = e * 5 * BN + pad(p);
      T u[5];
      T* v0 = V + o;
#pragma unroll
      for (int c = 0; c < 5; ++c) u[c] = ug(o + c * BN, e * 5 + c);
      const SideState<T> s = side_state(u, ph);
      if (GEO == GEO_AFFINE) {
        // reference derivatives; 1/h_j enters with 1/rho and with the flux constants
        T gu[3][3], ge[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const T* g = v0 + j * VS;
          const T r = kc.hinv[j] * s.rinv, g0 = g[0];
#pragma unroll
          for (int i = 0; i < 3; ++i) gu[i][j] = (g[(1 + i) * BN] - s.v[i] * g0) * r;
          ge[j] = (g[4 * BN] - s.E * g0) * r - (s.v[0] * gu[0][j] + s.v[1] * gu[1][j] + s.v[2] * gu[2][j]);
        }
        const T div = T(2) / T(3) * (gu[0][0] + gu[1][1] + gu[2][2]);
        const T s01 = gu[0][1] + gu[1][0], s02 = gu[0][2] + gu[2][0], s12 = gu[1][2] + gu[2][1];
        const T S[3][3] = {{T(2) * gu[0][0] - div, s01, s02}, {s01, T(2) * gu[1][1] - div, s12},
                           {s02, s12, T(2) * gu[2][2] - div}};
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          T* f = v0 + b * VS;
          const T w = -kc.muh[b];
          const T t0 = w * S[b][0], t1 = w * S[b][1], t2 = w * S[b][2];
          f[0] = T(0);
          f[BN] = see(1, t0);
          f[2 * BN] = see(2, t1);
          f[3 * BN] = see(3, t2);
          f[4 * BN] = see(4, t0 * s.v[0] + t1 * s.v[1] + t2 * s.v[2] - kc.lamh[b] * ge[b]);
        }
      } else {
        T Jd[9], G[5][3];
        const T* g = static_cast<const T*>(kp.gcv) + (size_t)(e0 + e) * 10 * N3 + p;
#pragma unroll
        for (int m = 0; m < 9; ++m) Jd[m] = g[m * N3];
#pragma unroll
        for (int c = 0; c < 5; ++c) {
          const T g0 = v0[c * BN], g1 = v0[VS + c * BN], g2 = v0[2 * VS + c * BN];
#pragma unroll
          for (int a = 0; a < 3; ++a) G[c][a] = Jd[a] * g0 + Jd[3 + a] * g1 + Jd[6 + a] * g2;
        }
        const T dj = -g[9 * N3];
#pragma unroll
        for (int m = 0; m < 9; ++m) Jd[m] *= dj;
        T gu[3][3];
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int j = 0; j < 3; ++j) gu[i][j] = (G[1 + i][j] - s.v[i] * G[0][j]) * s.rinv;
        const T div = T(2) / T(3) * (gu[0][0] + gu[1][1] + gu[2][2]);
        T t[3][3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          t[i][i] = ph.mu * (T(2) * gu[i][i] - div);
#pragma unroll
          for (int j = i + 1; j < 3; ++j) t[i][j] = t[j][i] = ph.mu * (gu[i][j] + gu[j][i]);
        }
        T q[3];
#pragma unroll
        for (int j = 0; j < 3; ++j)
          q[j] = t[0][j] * s.v[0] + t[1][j] * s.v[1] + t[2][j] * s.v[2] +
                 ph.lam_cv * ((G[4][j] - s.E * G[0][j]) * s.rinv -
                              (s.v[0] * gu[0][j] + s.v[1] * gu[1][j] + s.v[2] * gu[2][j]));
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          T* f = v0 + b * VS;
          const T j0 = Jd[3 * b], j1 = Jd[3 * b + 1], j2 = Jd[3 * b + 2];
          f[0] = T(0);
#pragma unroll
          for (int i = 0; i < 3; ++i) f[(1 + i) * BN] = see(1 + i, j0 * t[i][0] + j1 * t[i][1] + j2 * t[i][2]);
          f[4 * BN] = see(4, j0 * q[0] + j1 * q[1] + j2 * q[2]);
        }
      }
    }
  }
  if constexpr (FX) {
    if (visc && pe < nb) block_max<32>(exV + pe * 5, 1, 0, mag);
    fixB = conv && fixA && blocks_ok(exC, 5 * CB);
    if (fixB) {
      chain<1, QC, QC, -1, FROM_DOUBLE, TO_INT, QC2>(F0, F0, tb.eDcW, nbl * QC * QC, exC, 0, 2);
      chain<QC, QC, QC, -1, FROM_DOUBLE, TO_INT, QC2>(F1, F1, tb.eDcW, nbl * QC, exC, 0, 2);
      chain<QC * QC, QC, QC, -1, FROM_DOUBLE, TO_INT, QC2>(F2, F2, tb.eDcW, nbl, exC, 0, 2);
    }
  }
  if (conv && !fixB) {
    sw<T, 0, QC, QC, QC, QC, -1, PQ, PQ>(F0, F0, tb.eDcW, nbl);
    sw<T, 1, QC, QC, QC, QC, -1, PQ, PQ>(F1, F1, tb.eDcW, nbl);
    sw<T, 2, QC, QC, QC, QC, -1, PQ, PQ>(F2, F2, tb.eDcW, nbl);
  }
  __syncthreads();
  // 6-8. projection of the summed convective parts onto the l_g; D~ and face shares of the viscous arrays
  int gF = 0;  // exponent after the lift over the viscous fluxes' and shares'
  if constexpr (FX) {
    fixL = blocks_ok(exV, 5 * CB);
    fixR = fixB && fixL && GEO == GEO_AFFINE && !force && kp.out_mode != 0;
    gF = chain_gain(tb.eLift, 2);
    fixL = fixL && (fixR || GEO == GEO_STORED || force || kp.out_mode == 0);  // (else the summed S^-1 sweep takes doubles)
    if (fixB) {
      chain<QC * QC, QC, N, 1, FROM_SUM, TO_DOUBLE, QC2, 0, 0, PC>(F0, F0, tb.ePc, nbl, exC, chain_gain(tb.eDcW, 2), 0,
                                                                   CB * 5 * S::F, 1 << 30, exP);
    }
    if (fixL)
      chain_lift<N>(V, FBc, tb.eLift, nb, visc, VS, exV);
    else
      lift_fp64<N>(V, FBc, tb.eLift, nb, visc, VS);
  } else {
    lift_body<T, N, 0>(V, FBc, tb.eLift, nb, visc);
    lift_body<T, N, 1>(V + VS, FBc, tb.eLift, nb, visc);
    lift_body<T, N, 2>(V + 2 * VS, FBc, tb.eLift, nb, visc);
  }
  if (conv && !fixB) sw<T, 2, QC, QC, QC, N, 1, PQ, PQ, 3, false, 0, BQ>(F0, F0, tb.ePc, nbl, CB * 5 * S::F);
  __syncthreads();
  if constexpr (FX) {
    if (fixB) {
      // exP and exR need no check of their own: the fluxes lie in 2^-723..2^677 (fx_exp_ok), D~, P and S^-1 raise that by
      // less than 2^20, and a sum that cancels keeps at least one of its 61 bits or is zero, so that each of the three
      // results loses at most 64 bits: all exponents stay within the normal range (biased 100 to 1720)
      chain<QC, QC, N, 1, FROM_DOUBLE, TO_INT, N * QC, N, PC>(F0, F1, tb.ePc, nbl * N, exP, 0);
      __syncthreads();
      chain<1, QC, N, 1, FROM_INT, TO_DOUBLE, N2>(F1, F2, tb.ePc, nbl * N2, exP, chain_gain(tb.ePc));
    }
  }
  if (conv && !fixB) {
    sw<T, 1, QC, QC, N, N, 1, PQ, P1, 1, false, BQ>(F0, F1, tb.ePc, nbl);
    __syncthreads();
    sw<T, 0, QC, N, N, N, 1, P1, PN>(F1, F2, tb.ePc, nbl);
  }
  if (!conv)
    for (int i = threadIdx.x; i < nbl * BN; i += NTH) F2[i] = T(0);
  __syncthreads();
  // 9-11. M^-1 in the l_g basis is a scaling by 1/|J| (affine: in the flux scales); S^-1 back to the nodes
  T* sr = F2;
  const Eo<T> eBack = kp.out_mode == 0 ? tb.eSvT : tb.eSmi;
  int back = 0;  // the chain back to the nodes starts from the pass below
  if constexpr (FX) {
    if (fixR) chain_sum<N>(V, VS, F2, F1, tb.eSmi, nbl * N2, exV, gF, exP, 2 * chain_gain(tb.ePc), exR);
  }
  if (fixR) {
  } else if (GEO == GEO_AFFINE && !force && kp.out_mode != 0) {
    sw<T, 0, N, N, N, N, 1, PN, PN, 3, true>(V, F1, tb.eSmi, nbl, VS, F2);
  } else {
    for (int i = threadIdx.x; (FX ? i & ~31 : i) < nvals; i += NTH) {  // (FP64: whole warps, for the maxima)
      uint32_t m[1] = {0};
      if (!FX || i < nvals) {
        const int p = i % N3, e = i / (5 * N3), c = (i / N3) % 5;
        const int ip = pad(i);
        T r;
        if (FX && fixL) {
          const int64_t* v = reinterpret_cast<const int64_t*>(V) + ip;
          r = F2[ip] + T(fx_store(v[0] + v[VS] + v[2 * VS], fx_exp(exV[i / N3]) + gF + 3));
        } else {
          r = F2[ip] + (V[ip] + (V[VS + ip] + V[2 * VS + ip]));
        }
        if (kp.out_mode == 0) {
          const T w = tb.wm[p % N] * tb.wm[(p / N) % N] * tb.wm[p / N2];
          r *= GEO == GEO_AFFINE ? -w * kc.detJ : -w;
        } else {
          if (GEO == GEO_STORED) r *= rcp_of(static_cast<const T*>(kp.gm)[(size_t)(e0 + e) * N3 + p]);
          if (force && c > 0) {
            const int g = e * 5 * BN + pad(p), b = e * 5;
            r += c < 4 ? kc.bf[c - 1]
                       : (kc.bf[0] * ug(g + BN, b + 1) + kc.bf[1] * ug(g + 2 * BN, b + 2) + kc.bf[2] * ug(g + 3 * BN, b + 3)) *
                             rcp_of(ph.rho_r + ug(g, b));
          }
        }
        F0[ip] = r;
        if constexpr (FX) m[0] = fx_mag(r);
      }
      if constexpr (FX) block_max<N3>(exR, 0, min(i, nvals - 1) / N3, m);
    }
    __syncthreads();
    if constexpr (FX) {
      fixR = blocks_ok(exR, 5 * CB);
      if (fixR) chain<1, N, N, 1, FROM_DOUBLE, TO_INT, N2>(F0, F1, eBack, nbl * N2, exR, 0);
      back = 1;
    }
    if (!fixR) sw<T, 0, N, N, N, N, 1, PN, PN>(F0, F1, eBack, nbl);
  }
  __syncthreads();
  if constexpr (FX) {
    if (fixR && back) {
      chain<N, N, N, 1, FROM_INT, TO_INT, N2>(F1, F0, eBack, nbl * N, exR, 0);
      __syncthreads();
      chain<N2, N, N, 1, FROM_INT, TO_DOUBLE, N2>(F0, sr, eBack, nbl, exR, 2 * chain_gain(eBack));
    } else if (fixR) {
      chain<N, N, N, 1, FROM_DOUBLE, TO_INT, N2>(F1, F0, tb.eSmi, nbl * N, exR, 0);
      __syncthreads();
      chain<N2, N, N, 1, FROM_INT, TO_DOUBLE, N2>(F0, sr, tb.eSmi, nbl, exR, chain_gain(tb.eSmi));
    }
  }
  if (!fixR) {
    sw<T, 1, N, N, N, N, 1, PN, PN>(F1, F0, eBack, nbl);
    __syncthreads();
    sw<T, 2, N, N, N, N, 1, PN, N2>(F0, sr, eBack, nbl);
  }
  __syncthreads();
  if (kp.out_mode == 2)
    stage_update<PER, N3>(kp, U, dU, Uout, sr, base, nvals, threadIdx.x, NTH);
  else
    for (int i = threadIdx.x; i < nvals; i += NTH) Rout[base + i] = sr[i];
}

// ---------------------------------------------------------------------------
// Face kernel.  Per face five component slots in the order (m_t1, rho, m_D, m_t2, rho E), so that the
// tangential derivatives an axis-aligned face needs (along t1: m_t1, rho, m_D; along t2: rho, m_D, m_t2) are
// contiguous; arrays are [slot][face][points].
// ---------------------------------------------------------------------------
template <int D>
__device__ __forceinline__ constexpr int slot_comp(int s) {
  constexpr int t1 = D == 0 ? 1 : 0, t2 = D == 2 ? 1 : 2;
  return s == 0 ? 1 + t1 : (s == 1 ? 0 : (s == 2 ? 1 + D : (s == 3 ? 1 + t2 : 4)));
}

template <int N, int QC>
struct CollFaceSizes {
  static constexpr int N2 = N * N, QC2 = QC * QC;
  static constexpr int VV = 4 * 5 * N2;        // traces: values and normal derivatives of both sides, nodal and then at
                                               // the viscous points; later the value and normal-gradient shares
  static constexpr int TT = 4 * 5 * N2;        // tangential derivatives, 2 directions x 2 sides; later gradient tests
  static constexpr int C0 = 2 * 5 * QC * N > 2 * 5 * N2 ? 2 * 5 * QC * N : 2 * 5 * N2;
  static constexpr int C1 = 2 * 5 * QC2;
  static constexpr int PER_FACE = VV + TT + C0 + C1;
};
template <typename T, int N, int QC, int QV>
constexpr size_t coll_face_smem(int fb) {
  return ((size_t)table_elems<T, N, QC, QV>() + (size_t)fb * (CollFaceSizes<N, QC>::PER_FACE + 1)) * sizeof(T) +
         (3 + (sizeof(T) == 8 ? 20 : 0)) * fb * sizeof(int) + 64;
}
// Faces per CTA: up to 8, as long as four CTAs fit an SM (56 KB each).
template <typename T, int N, int QC, int QV>
constexpr int coll_faces() {
  int fb = 8;
  while (fb > 1 && coll_face_smem<T, N, QC, QV>(fb) > 56 * 1024) --fb;
  return fb;
}
// (FP32 at k = 4, 5: 256 threads for the larger faces, 1.10 -> 0.89 ms at 40^3, k = 5)
template <typename T, int N>
constexpr int coll_face_threads() {
  return sizeof(T) == 4 && N >= 5 ? 256 : 128;
}
// Resident CTAs that the registers have to allow: FP64 four, with general metrics three (168 registers; without the bound
// they are two and the kernel a third slower); FP32 0, no bound.
template <typename T, int GEO>
constexpr int coll_face_ctas() {
  return sizeof(T) == 4 ? 0 : (GEO == GEO_AFFINE ? 4 : 3);
}

template <typename T, int N, int QC, int QV, int FB_, int D, int GEO>
__device__ __forceinline__ void coll_face_terms(const double* U, const T* Ud, const int* eo,
                                                const int* en, const int* oc, const T* tau_f, T* sm, const Tab<T>& tb,
                                                const KParams& kp, const PhysT<T>& ph, int nb, int s, T* FBuf,
                                                uint32_t* ex) {
  using Z = CollFaceSizes<N, QC>;
  constexpr int N2 = N * N, N3 = N2 * N, QC2 = QC * QC, NTH = coll_face_threads<T, N>();
  constexpr int t1 = D == 0 ? 1 : 0, t2 = D == 2 ? 1 : 2;
  constexpr bool AFF = GEO == GEO_AFFINE;
  const KConst<T>& kc = kconst<T>(kp);
  const int f = 2 * D + s, fo = 2 * D + (1 - s);
  const T* dlm = s ? tb.dl1 : tb.dl0;
  const T* dlp = s ? tb.dl0 : tb.dl1;
  const int nf = nb * N2, nl = 5 * nf;  // values per slot and per array
  T* VV = sm;                      // [Lm, Lp, Dm, Dp][5][nb][N2]
  T* TT = VV + FB_ * Z::VV;        // [t1 m, t1 p, t2 m, t2 p][5 (3 used if AFF)][nb][N2]
  T* C0 = TT + FB_ * Z::TT;
  T* C1 = C0 + FB_ * Z::C0;        // [m, p][5][nb][QC2]; later the convective share [5][nb][N2]
  const bool conv = kp.conv != 0, visc = kp.visc != 0;
  constexpr bool FX = sizeof(T) == 8;  // integer chains
  constexpr int NTT = AFF ? 3 : 5;     // tested components of a tangential direction
  // FP64: maxima of the blocks (slot, face), both sides together: of the traces, of the normal derivatives, of the
  // convective flux and of the tangential gradient tests.  (On an axis-aligned face m_t1 along t1 and m_t2 along t2 share
  // a block: both are -2/3 mu g_D / rho, times 1/h_t1 and 1/h_t2, so that the smaller loses the bits of that aspect ratio,
  // of 61; its row's own second derivatives lose twice as many to rounding, of 53.)
  uint32_t *exL = ex, *exD = exL + 5 * FB_, *exC = exD + 5 * FB_, *exT = exC + 5 * FB_;
  auto see = [&](uint32_t& m, T v) {
    if constexpr (FX) m = max(m, fx_mag(v));
    return v;
  };
  // traces along the normal lines, from global memory
  for (int idx = threadIdx.x; idx < nl; idx += NTH) {
    const int sl = idx / nf, r = idx - sl * nf, e = r / N2, j = r - e * N2;
    const int c = slot_comp<D>(sl);
    const int q0 = face_node<N>(D, 0, j % N, j / N);
    constexpr int st = D == 0 ? 1 : (D == 1 ? N : N2);
    const size_t om = ((size_t)eo[e] * 5 + c) * N3 + q0;
    const int eq = en[e];
    size_t op = ((size_t)(eq < 0 ? 0 : eq) * 5 + c) * N3;
    int qs = st;
    if (oc && eq >= 0) {
      // rotated-frame meshes: the normal line is a line of the other cell too, at a constant stride from its
      // reoriented first node
      const int r0 = frame_node<N>(oc[e], q0);
      qs = frame_node<N>(oc[e], q0 + st) - r0;
      op += r0;
    } else {
      op += q0;
    }
    T a[N], b[N];
    if (Ud) {
#pragma unroll
      for (int i = 0; i < N; ++i) {
        a[i] = Ud[om + i * st];
        b[i] = eq < 0 ? T(0) : Ud[op + i * qs];
      }
    } else {
      double ud[N], un[N];  // (all loads of the line before the first conversion)
#pragma unroll
      for (int i = 0; i < N; ++i) {
        ud[i] = U[om + i * st];
        un[i] = U[eq < 0 ? om : op + i * qs];
      }
#pragma unroll
      for (int i = 0; i < N; ++i) {
        a[i] = dev_value<T>(kp, ud[i], c);
        b[i] = eq < 0 ? T(0) : dev_value<T>(kp, un[i], c);
      }
    }
    T dm, dp;
    if constexpr (FX) {
      T y[2], z[2];
      line_apply<T, N, 2, -1>(tb.eDl, a, y);
      line_apply<T, N, 2, -1>(tb.eDl, b, z);
      dm = s ? y[1] : y[0];
      dp = s ? z[0] : z[1];
    } else {
      dm = dp = T(0);
#pragma unroll
      for (int i = 0; i < N; ++i) {
        dm += dlm[i] * a[i];
        dp += dlp[i] * b[i];
      }
    }
    const T vm = s ? a[N - 1] : a[0], vp = s ? b[0] : b[N - 1];
    VV[idx] = vm;
    VV[nl + idx] = vp;
    VV[2 * nl + idx] = dm;
    VV[3 * nl + idx] = dp;
    if constexpr (FX) {
      const uint32_t m[2] = {max(fx_mag(vm), fx_mag(vp)), max(fx_mag(dm), fx_mag(dp))};
      block_max<1>(exL, 5 * FB_, idx / N2, m);
    }
  }
  __syncthreads();
  bool fixA = false;
  int gS = 0;
  if constexpr (FX) {
    fixA = blocks_ok(exL, 10 * FB_);
    if (fixA) {
      gS = chain_gain(tb.eSm);
      if (conv) chain<1, N, QC, 1, FROM_DOUBLE, TO_INT, N>(VV, C0, tb.eSc, 2 * 5 * nb * N, exL, 0, 0, 0, 5 * nb);
      if (visc) {
        chain<1, N, N, 1, FROM_DOUBLE, TO_INT, N>(VV, TT, tb.eSm, 2 * 5 * nb * N, exL, 0, 0, 0, 5 * nb);
        chain<1, N, N, 1, FROM_DOUBLE, TO_INT, N>(VV + 2 * nl, TT + 2 * nl, tb.eSm, 2 * 5 * nb * N, exD, 0, 0, 0, 5 * nb);
      }
    }
  }
  if (!fixA) {
    if (conv) sw<T, 0, N, N, 1, QC, 1>(VV, C0, tb.eSc, 10 * nb);
    if (visc) sw<T, 0, N, N, 1, N, 1>(VV, TT, tb.eSm, 20 * nb);
  }
  __syncthreads();
  if constexpr (FX) {
    if (fixA) {
      if (conv) chain<QC, N, QC, 1, FROM_INT, TO_DOUBLE, QC>(C0, C1, tb.eSc, 2 * 5 * nb, exL, chain_gain(tb.eSc), 0, 0, 5 * nb);
      if (visc) {
        chain<N, N, N, 1, FROM_INT, TO_INT, N>(TT, VV, tb.eSm, 2 * 5 * nb, exL, 0);
        chain<N, N, N, 1, FROM_INT, TO_DOUBLE, N>(TT + 2 * nl, VV + 2 * nl, tb.eSm, 2 * 5 * nb, exD, gS, 0, 0, 5 * nb);
      }
      gS *= 2;
    }
  }
  if (!fixA) {
    if (conv) sw<T, 1, QC, N, 1, QC, 1>(C0, C1, tb.eSc, 10 * nb);
    if (visc) sw<T, 1, N, N, 1, N, 1>(TT, VV, tb.eSm, 20 * nb);
  }
  __syncthreads();
  // convective flux (point arithmetic); tangential derivatives (sweeps)
  if (conv) {
    const int nc = nb * QC2;
    for (int idx = threadIdx.x; idx < nc; idx += NTH) {
      uint32_t mC[5] = {0, 0, 0, 0, 0};
      const int e = idx / QC2, p = idx - e * QC2;
      T um[5], up[5], fm[5], fp[5], n[3] = {T(0), T(0), T(0)}, w;
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        um[slot_comp<D>(q)] = C1[q * nc + idx];
        up[slot_comp<D>(q)] = C1[(5 + q) * nc + idx];
      }
      if (en[e] < 0) wall_ghost(um, ph, up);
      if (AFF) {
        w = T(-0.5) * kc.hinv[D];
      } else {
        const T* g = static_cast<const T*>(kp.gfc) + ((size_t)eo[e] * 6 + f) * 13 * QC2 + p;
        n[0] = g[9 * QC2];
        n[1] = g[10 * QC2];
        n[2] = g[11 * QC2];
        w = T(-0.5) * g[12 * QC2];
      }
      T lm, lp;
      const T ws = AFF && !s ? -w : w;
      llf_side<T, D, AFF>(um, n, ws, ph, fm, lm);
      llf_side<T, D, AFF>(up, n, ws, ph, fp, lp);
      const T lam = w * (lm > lp ? lm : lp);
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        const int c = slot_comp<D>(q);
        C1[q * nc + idx] = see(mC[q], fm[c] + fp[c] + lam * (um[c] - up[c]));
      }
      if constexpr (FX) block_max<1>(exC, nb, e, mC);
    }
  }
  if constexpr (FX) {
    if (visc && fixA) {
#pragma unroll
      for (int sd = 0; sd < 2; ++sd) {
        const int o = sd * nl;
        if (AFF) {
          chain<1, N, N, -1, FROM_INT, TO_DOUBLE, N>(VV + o, TT + o, tb.eDv, 3 * nb * N, exL, gS);
          chain<N, N, N, -1, FROM_INT, TO_DOUBLE, N>(VV + o + nf, TT + 2 * nl + o, tb.eDv, 3 * nb, exL + nb, gS);
        } else {
          chain<1, N, N, -1, FROM_INT, TO_DOUBLE, N>(VV + o, TT + o, tb.eDv, 5 * nb * N, exL, gS);
          chain<N, N, N, -1, FROM_INT, TO_DOUBLE, N>(VV + o, TT + 2 * nl + o, tb.eDv, 5 * nb, exL, gS);
        }
      }
    }
  }
  if (visc && !fixA) {
    if (AFF) {
#pragma unroll
      for (int sd = 0; sd < 2; ++sd) {
        sw<T, 0, N, N, 1, N, -1>(VV + sd * nl, TT + sd * nl, tb.eDv, 3 * nb);
        sw<T, 1, N, N, 1, N, -1>(VV + sd * nl + nf, TT + (2 + sd) * nl, tb.eDv, 3 * nb);
      }
    } else {
      sw<T, 0, N, N, 1, N, -1>(VV, TT, tb.eDv, 10 * nb);
      sw<T, 1, N, N, 1, N, -1>(VV, TT + 2 * nl, tb.eDv, 10 * nb);
    }
  }
  __syncthreads();
  // viscous fluxes (point arithmetic); projection of the convective flux (sweeps).  Shares are of -F.
  if (visc) {
    for (int idx = threadIdx.x; idx < nf; idx += NTH) {
      uint32_t mT[NTT] = {};
      const int e = idx / N2, p = idx - e * N2;
      const bool wall = en[e] < 0;
      T um[5], up[5], jmp[5];
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        T a = VV[q * nf + idx], b = VV[nl + q * nf + idx];
        if constexpr (FX) {
          if (fixA) {
            const int X = fx_exp(exL[q * nb + e]) + gS + 3;
            a = fx_store(__double_as_longlong(a), X);
            b = fx_store(__double_as_longlong(b), X);
          }
        }
        um[slot_comp<D>(q)] = a;
        up[slot_comp<D>(q)] = b;
      }
      if (wall) wall_ghost(um, ph, up);
      const SideState<T> sm_ = side_state(um, ph), sp_ = side_state(up, ph);
      const T tau = tau_f[e];
#pragma unroll
      for (int c = 0; c < 5; ++c) jmp[c] = um[c] - up[c];
      T fm[4], fp[4];
      if (AFF) {
        const T hd = kc.hinv[D];
        T* T1m = TT + idx;
        T* T1p = T1m + nl;
        T* T2m = T1p + nl;
        T* T2p = T2m + nl;
        T gm[5], gp[5];
#pragma unroll
        for (int q = 0; q < 5; ++q) {
          gm[slot_comp<D>(q)] = VV[2 * nl + q * nf + idx];
          gp[slot_comp<D>(q)] = VV[3 * nl + q * nf + idx];
        }
        visc_normal<T, D>(sm_, gm, T1m[nf], T1m[2 * nf], T1m[0], T2m[0], T2m[nf], T2m[2 * nf], kc, fm);
        if (wall)  // grad U+ = grad U-, at the ghost state
          visc_normal<T, D>(sp_, gm, T1m[nf], T1m[2 * nf], T1m[0], T2m[0], T2m[nf], T2m[2 * nf], kc, fp);
        else
          visc_normal<T, D>(sp_, gp, T1p[nf], T1p[2 * nf], T1p[0], T2p[0], T2p[nf], T2p[2 * nf], kc, fp);
        // value share (own side): (V, Q*.n), Q*.n = {{F_v}}.n - tau [[U]]; the other side's is the negative
        const T wv = s ? T(0.5) * hd : T(-0.5) * hd, wt = hd * tau;
        const int fs[5] = {1, -1, 0, 2, 3};  // slot -> entry of fm
#pragma unroll
        for (int q = 0; q < 5; ++q) {
          const T t = -wt * jmp[slot_comp<D>(q)];
          VV[q * nf + idx] = fs[q] < 0 ? t : t + wv * (fm[fs[q] < 0 ? 0 : fs[q]] + fp[fs[q] < 0 ? 0 : fs[q]]);
        }
        // +1/2 (grad V, F_v(U, [[U]])), [[U]] = sgn jmp (x) e_D
        if (!s) {
#pragma unroll
          for (int c = 0; c < 5; ++c) jmp[c] = -jmp[c];
        }
        T a[4], b1[3], b2[3];
        visc_jump<T, D>(sm_, jmp, kc, a, b1, b2);
        VV[2 * nl + idx] = a[1];
        VV[2 * nl + nf + idx] = T(0);
        VV[2 * nl + 2 * nf + idx] = a[0];
        VV[2 * nl + 3 * nf + idx] = a[2];
        VV[2 * nl + 4 * nf + idx] = a[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          T1m[i * nf] = see(mT[i], b1[i]);
          T2m[i * nf] = see(mT[i], b2[i]);
        }
        if (!wall) visc_jump<T, D>(sp_, jmp, kc, a, b1, b2);
        VV[3 * nl + idx] = a[1];
        VV[3 * nl + nf + idx] = T(0);
        VV[3 * nl + 2 * nf + idx] = a[0];
        VV[3 * nl + 3 * nf + idx] = a[2];
        VV[3 * nl + 4 * nf + idx] = a[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          T1p[i * nf] = see(mT[i], b1[i]);
          T2p[i * nf] = see(mT[i], b2[i]);
        }
      } else {
        const T* g = static_cast<const T*>(kp.gfv) + ((size_t)eo[e] * 6 + f) * 13 * N2 + p;
        T Jm[9], Jp[9], n[3];
#pragma unroll
        for (int m = 0; m < 9; ++m) Jm[m] = g[m * N2];
        n[0] = g[9 * N2];
        n[1] = g[10 * N2];
        n[2] = g[11 * N2];
        const T dA = g[12 * N2];
        if (!wall && oc) {
          frame_face_jinv<T, N>(static_cast<const T*>(kp.gfv), en[e], oc[e], D, s, p, Jp);
        } else {
          const T* gp = wall ? g : static_cast<const T*>(kp.gfv) + ((size_t)en[e] * 6 + fo) * 13 * N2 + p;
#pragma unroll
          for (int m = 0; m < 9; ++m) Jp[m] = gp[m * N2];
        }
        T G[5][3];
#pragma unroll
        for (int q = 0; q < 5; ++q) {
          const T a1 = TT[q * nf + idx], a2 = TT[2 * nl + q * nf + idx], ad = VV[2 * nl + q * nf + idx];
#pragma unroll
          for (int a = 0; a < 3; ++a) G[slot_comp<D>(q)][a] = Jm[3 * t1 + a] * a1 + Jm[3 * t2 + a] * a2 + Jm[3 * D + a] * ad;
        }
        visc_normal_any(sm_, G, n, ph, fm);
        if (!wall) {
#pragma unroll
          for (int q = 0; q < 5; ++q) {
            const T a1 = TT[nl + q * nf + idx], a2 = TT[3 * nl + q * nf + idx], ad = VV[3 * nl + q * nf + idx];
#pragma unroll
            for (int a = 0; a < 3; ++a) G[slot_comp<D>(q)][a] = Jp[3 * t1 + a] * a1 + Jp[3 * t2 + a] * a2 + Jp[3 * D + a] * ad;
          }
        }
        visc_normal_any(sp_, G, n, ph, fp);
        const T hw = T(0.5) * dA, wt = dA * tau;
#pragma unroll
        for (int q = 0; q < 5; ++q) {
          const int c = slot_comp<D>(q);
          const T t = -wt * jmp[c];
          VV[q * nf + idx] = c == 0 ? t : t + hw * (fm[c == 0 ? 0 : c - 1] + fp[c == 0 ? 0 : c - 1]);
        }
#pragma unroll
        for (int sd = 0; sd < 2; ++sd) {
          const SideState<T>& ss = sd ? sp_ : sm_;
          const T* J = sd ? Jp : Jm;
          const JumpFlux<T> jf = visc_jump_any(ss, jmp, n, ph);
          T* dst[3] = {TT + sd * nl + idx, TT + (2 + sd) * nl + idx, VV + (2 + sd) * nl + idx};
          const int row[3] = {t1, t2, D};
#pragma unroll
          for (int b = 0; b < 3; ++b) {
            T r[4];
            jump_row(jf, ss, n, J + 3 * row[b], hw, r);
#pragma unroll
            for (int q = 0; q < 5; ++q) {
              const int c = slot_comp<D>(q);
              const T v = c == 0 ? T(0) : r[c == 0 ? 0 : c - 1];
              dst[b][q * nf] = b < 2 ? see(mT[q], v) : v;
            }
          }
        }
      }
      if constexpr (FX) block_max<1>(exT, nb, e, mT);
    }
  }
  bool fixB = false, fixT = false;
  if constexpr (FX) {
    fixB = conv && blocks_ok(exC, 5 * nb);
    if (fixB) chain<QC, QC, N, 1, FROM_DOUBLE, TO_INT, QC>(C1, C0, tb.ePc, 5 * nb, exC, 0);
  }
  if (conv && !fixB) sw<T, 1, QC, QC, 1, N, 1>(C1, C0, tb.ePc, 5 * nb);
  __syncthreads();
  // tangential gradient tests, in place; the convective share
  int gT = 0;
  if constexpr (FX) {
    fixT = visc && blocks_ok(exT, NTT * nb);
    if (fixT) {
      gT = chain_gain(tb.eDvW, 1);
#pragma unroll
      for (int sd = 0; sd < 2; ++sd) {
        double* t1a = TT + sd * nl;
        double* t2a = TT + (2 + sd) * nl;
        chain<1, N, N, -1, FROM_DOUBLE, TO_INT, N>(t1a, t1a, tb.eDvW, NTT * nb * N, exT, 0, 1);
        chain<N, N, N, -1, FROM_DOUBLE, TO_INT, N>(t2a, t2a, tb.eDvW, NTT * nb, exT, 0, 1);
      }
    }
    if (fixB) chain<1, QC, N, 1, FROM_INT, TO_DOUBLE, N>(C0, C1, tb.ePc, 5 * nb * N, exC, chain_gain(tb.ePc));
  }
  if (visc && !fixT) {
    if (AFF) {
#pragma unroll
      for (int sd = 0; sd < 2; ++sd) {
        sw<T, 0, N, N, 1, N, -1>(TT + sd * nl, TT + sd * nl, tb.eDvW, 3 * nb);
        sw<T, 1, N, N, 1, N, -1>(TT + (2 + sd) * nl, TT + (2 + sd) * nl, tb.eDvW, 3 * nb);
      }
    } else {
      sw<T, 0, N, N, 1, N, -1>(TT, TT, tb.eDvW, 10 * nb);
      sw<T, 1, N, N, 1, N, -1>(TT + 2 * nl, TT + 2 * nl, tb.eDvW, 10 * nb);
    }
  }
  if (conv && !fixB) sw<T, 0, QC, N, 1, N, 1>(C0, C1, tb.ePc, 5 * nb);
  __syncthreads();
  // shares of the own and the other cell
  for (int idx = threadIdx.x; idx < nl; idx += NTH) {
    const int sl = idx / nf, r = idx - sl * nf, e = r / N2, j = r - e * N2;
    const int c = slot_comp<D>(sl);
    T lm = T(0), lp = T(0), dm = T(0), dp = T(0);
    if (visc) {
      lm = VV[idx];
      lp = -lm;
      dm = VV[2 * nl + idx];
      dp = VV[3 * nl + idx];
      // tested entries of an axis-aligned face: along t1 (m_D, m_t1, rho E), along t2 (m_D, m_t2, rho E)
      const int k1 = !AFF ? sl : (sl == 2 ? 0 : (sl == 0 ? 1 : (sl == 4 ? 2 : -1)));
      const int k2 = !AFF ? sl : (sl == 2 ? 0 : (sl == 3 ? 1 : (sl == 4 ? 2 : -1)));
      bool done = false;
      if constexpr (FX) {
        if (fixT) {
          const int k = k1 < 0 ? k2 : k1;
          if (k >= 0) {
            const int64_t* t = reinterpret_cast<const int64_t*>(TT) + r;
            int64_t a = 0, b = 0;
            if (k1 >= 0) {
              a = t[k1 * nf];
              b = t[nl + k1 * nf];
            }
            if (k2 >= 0) {
              a += t[2 * nl + k2 * nf];
              b += t[3 * nl + k2 * nf];
            }
            const int X = fx_exp(exT[k * nb + e]) + gT + 3;
            lm += fx_store(a, X);
            lp += fx_store(b, X);
          }
          done = true;
        }
      }
      if (!done) {
        if (k1 >= 0) {
          lm += TT[k1 * nf + r];
          lp += TT[nl + k1 * nf + r];
        }
        if (k2 >= 0) {
          lm += TT[2 * nl + k2 * nf + r];
          lp += TT[3 * nl + k2 * nf + r];
        }
      }
    }
    if (conv) {
      const T l = C1[idx];
      lm += l;
      lp -= l;
    }
    T* po = FBuf + ((size_t)eo[e] * 6 + f) * 10 * N2 + c * N2 + j;
    po[0] = lm;
    po[5 * N2] = dm;
    if (en[e] >= 0) {
      int fw = fo, jw = j;
      T dsg = T(1);
      if (oc) {
        // the other cell's face point of this face point, in its own frame
        int dn, refl, sn;
        frame_facing(oc[e], D, s, dn, refl, sn);
        const int q = frame_node<N>(oc[e], face_node<N>(D, s ? 0 : N - 1, j % N, j / N));
        const int q0 = q % N, q1 = (q / N) % N, q2 = q / N2;
        fw = 2 * dn + sn;
        jw = dn == 0 ? q1 + N * q2 : (dn == 1 ? q0 + N * q2 : q0 + N * q1);
        dsg = refl ? T(-1) : T(1);
      }
      T* pn = FBuf + ((size_t)en[e] * 6 + fw) * 10 * N2 + c * N2 + jw;
      pn[0] = lp;
      pn[5 * N2] = dsg * dp;
    }
  }
}

// blockIdx.y = direction; blocks as dg_face_kernel.
template <typename T, int N, int QC, int QV, int FB_, int GEO>
__global__ void __launch_bounds__(coll_face_threads<T, N>(), coll_face_ctas<T, GEO>()) dg_coll_face_kernel(const KParams kp,
                                                                              const double* U, T* FBuf) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* stab = reinterpret_cast<T*>(smem_raw);
  T* sm = stab + table_elems<T, N, QC, QV>();
  T* tau_f = sm + FB_ * CollFaceSizes<N, QC>::PER_FACE;
  int* eo = reinterpret_cast<int*>(tau_f + FB_);
  int* en = eo + FB_;
  int* oc = en + FB_;
  uint32_t* ex = reinterpret_cast<uint32_t*>(oc + FB_);
  for (int i = threadIdx.x; sizeof(T) == 8 && i < 20 * FB_; i += blockDim.x) ex[i] = 0;
  const int d = blockIdx.y;
  int s, nb;
  const Tab<T> tb = load_tables<T, N, QC, QV>(static_cast<const T*>(kp.tables), stab);
  const PhysT<T> ph = make_phys<T>(kp);
  wait_for_predecessor();
  if (!face_batch<FB_>(kp, d, s, nb, eo, en, oc, tau_f)) return;
  __syncthreads();
  const T* Ud = static_cast<const T*>(kp.Udev);
  const int* ocp = kp.flist ? oc : nullptr;
  if (d == 0)
    coll_face_terms<T, N, QC, QV, FB_, 0, GEO>(U, Ud, eo, en, ocp, tau_f, sm, tb, kp, ph, nb, s, FBuf, ex);
  else if (d == 1)
    coll_face_terms<T, N, QC, QV, FB_, 1, GEO>(U, Ud, eo, en, ocp, tau_f, sm, tb, kp, ph, nb, s, FBuf, ex);
  else
    coll_face_terms<T, N, QC, QV, FB_, 2, GEO>(U, Ud, eo, en, ocp, tau_f, sm, tb, kp, ph, nb, s, FBuf, ex);
}

// Where the collocation kernels exist; the face-centric organisation then runs them (face and cell kernel share the face
// buffer's basis, so both follow this rule).
template <typename T, int N, int QC, int QV, int GEO>
constexpr bool coll_ok() {
  return QV == N && coll_rule(N, QV) && GEO != GEO_FLY && coll_cell_smem<T, N, QC, QV, 1>() <= 227 * 1024;
}

// Small meshes: half the cells or faces per CTA with as many threads, so that the phases of a CTA get shorter, as long as
// all those CTAs are resident at once; beyond that the second, partly empty wave costs more than the shorter phases give
// (L(U), half batches up to twice that size -> this rule: FP64 k = 3 9^3 cells 121 -> 105 us, k = 1 10^3 67 -> 45 us; FP32
// k = 5 10^3 54 -> 42 us).
template <typename T, int N, int QC, int QV, int CB, int GEO>
int launch_coll_cell_cb(const KParams& kp, bool only_one_wave, const double* U, void* Rout, void* dU, double* Uout,
                        cudaStream_t st) {
  constexpr size_t smem = coll_cell_smem<T, N, QC, QV, CB>();
  static_assert(smem <= 227 * 1024, "cell kernel shared memory");
  auto k = dg_coll_cell_kernel<T, N, QC, QV, CB, GEO>;
  constexpr int threads = coll_threads<T, N, QC, QV>();
  static bool attr[kMaxDevices] = {};
  static int per_sm[kMaxDevices] = {};
  if (smem_attr_once(k, smem, attr)) return -1;
  const int ctas = (kp.Nc + CB - 1) / CB;
  if (only_one_wave && !one_wave(k, threads, smem, ctas, per_sm)) return 1;
  return launch_after(k, dim3(ctas), threads, smem, st, kp, U, static_cast<T*>(Rout), static_cast<T*>(dU), Uout);
}
template <typename T, int N, int QC, int QV, int GEO>
int launch_coll_cell(const KParams& kp, const double* U, void* Rout, void* dU, double* Uout, cudaStream_t st) {
  constexpr int CB = coll_cells<T, N, QC, QV>();
  if constexpr (CB > 1) {
    const int r = launch_coll_cell_cb<T, N, QC, QV, CB / 2, GEO>(kp, true, U, Rout, dU, Uout, st);
    if (r <= 0) return r;
  }
  return launch_coll_cell_cb<T, N, QC, QV, CB, GEO>(kp, false, U, Rout, dU, Uout, st);
}

template <typename T, int N, int QC, int QV, int FB_, int GEO>
int launch_coll_faces_fb(const KParams& kp, bool only_one_wave, const double* U, void* FB, cudaStream_t st) {
  constexpr size_t smem = coll_face_smem<T, N, QC, QV>(FB_);
  static_assert(smem <= 227 * 1024, "face kernel shared memory");
  auto k = dg_coll_face_kernel<T, N, QC, QV, FB_, GEO>;
  constexpr int threads = coll_face_threads<T, N>();
  static bool attr[kMaxDevices] = {};
  static int per_sm[kMaxDevices] = {};
  if (smem_attr_once(k, smem, attr)) return -1;
  const int blocks = face_blocks(kp, FB_);
  if (only_one_wave && !one_wave(k, threads, smem, 3ll * blocks, per_sm)) return 1;
  return launch_after(k, dim3(blocks, 3), threads, smem, st, kp, U, static_cast<T*>(FB));
}
template <typename T, int N, int QC, int QV, int GEO>
int launch_coll_faces(const KParams& kp, const double* U, void* FB, cudaStream_t st) {
  constexpr int FB_ = coll_faces<T, N, QC, QV>();
  if constexpr (FB_ > 1) {
    const int r = launch_coll_faces_fb<T, N, QC, QV, FB_ / 2, GEO>(kp, true, U, FB, st);
    if (r <= 0) return r;
  }
  return launch_coll_faces_fb<T, N, QC, QV, FB_, GEO>(kp, false, U, FB, st);
}

}  // namespace dgcns
