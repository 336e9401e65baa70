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
// Measured per launch, against the kernels that test with the LGL basis (face / cell + stage kernel):
// FP64 TGV 64^3, k = 3: 24.6 -> 13.4 / 21.2 -> 14.9 ms; 40^3, k = 5: 14.9 -> 10.9 / 25.7 -> 15.2 ms;
// FP32 40^3, k = 5: 1.36 -> 1.12 / 2.51 -> 1.30 ms; channel 32^3, k = 3: 0.36 -> 0.29 / 0.36 -> 0.26 ms;
// FP32 64^3, k = 3, cell + stage: 2.14 (register-resident tasks, one cell per CTA) -> 1.60 ms.
// Bound by: FP64 faces the FP64 pipe (64 % busy, 6,450 instructions a face); FP64 cells latency and
// instruction fetch (ALU 46 %, FP64 34 %, issue 43 %).
#pragma once
#include "dg_faces.cuh"
#include "dg_kernels.cuh"

namespace dgcns {

// ---------------------------------------------------------------------------
// Reciprocal and square root of the point fluxes.  FP64: the hardware's seed (about 2^-20) and one
// third-order step, r (1 + e + e^2) with e = 1 - x r (Householder's iteration; the error is e^3 and one
// rounding): 3 FP64 instructions where the division measured 8 on GB300.  Outside the seed's range (zero,
// denormal, huge, infinite, NaN) the division itself.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float rcp_of(float x) { return 1.f / x; }
__device__ __forceinline__ double rcp_of(double x) {
  const uint32_t h = (uint32_t)__double2hiint(x) & 0x7fffffffu;
  if (h - 0x01000000u > 0x7d000000u) return 1.0 / x;
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}
// sqrt(a), a >= 0: h = a y with y the seed of 1/sqrt(a), e = 1 - h y, h (1 + e/2 + 3 e^2/8).
__device__ __forceinline__ float sqrt_of(float a) { return sqrtf(a); }
__device__ __forceinline__ double sqrt_of(double a) {
  const uint32_t t = (uint32_t)__double2hiint(a);
  if (t - 0x01000000u > 0x7d000000u) return sqrt(a);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
  const double h = a * y;
  const double e = fma(-h, y, 1.0);
  return fma(h, fma(e, 0.375, 0.5) * e, h);
}

// ---------------------------------------------------------------------------
// Sweeps.  Lines of DIN values at stride n0 of contiguous arrays -> DOUT values; line l = (outer, inner)
// with inner < n0 starts at outer n0 DIN + inner.  NIN: the input is the sum of NIN arrays ks apart (and of
// `extra` when EX).  OG > 0: OG consecutive outers form a block, blocks IBS apart in the input.  OBS > 0:
// outers are OBS apart in the output (an in-place sweep that keeps its block stride).
// ---------------------------------------------------------------------------
template <typename T, int DIN, int DOUT, int SYM, int NIN, bool EX, int OG, int IBS, int OBS>
__device__ __forceinline__ void lines_body(const T* in, int ks, const T* extra, T* out, Eo<T> E, int nlines, int n0,
                                           uint32_t magic, int rank, int stride) {
  for (int l = rank; l < nlines; l += stride) {
    int outer;
    if constexpr (sizeof(T) == 8)
      outer = n0 > 1 ? (int)__umulhi((uint32_t)l, magic) : l;
    else
      outer = l / n0;
    const int inner = l - outer * n0;
    const int ib = (OG > 0 ? (outer / (OG > 0 ? OG : 1)) * IBS + (outer % (OG > 0 ? OG : 1)) * n0 * DIN : outer * n0 * DIN) + inner;
    const int ob = (OBS > 0 ? outer * OBS : outer * n0 * DOUT) + inner;
    const T* ip = in + ib;
    T* op = out + ob;
    T y[DOUT];
    constexpr bool VIN = NIN == 1 && !EX && (DIN * sizeof(T)) % 16 == 0;
    constexpr bool VOUT = (DOUT * sizeof(T)) % 16 == 0;
    if constexpr (NIN + (EX ? 1 : 0) == 1) {
      T x[DIN];
      bool loaded = false;
      if constexpr (VIN) {
        // a line along x is contiguous: 16-byte accesses avoid the bank conflicts of threads reading
        // DIN-value lines at a DIN-value stride
        if (n0 == 1 && (reinterpret_cast<uintptr_t>(ip) & 15) == 0) {
          vec_load<T, DIN>(ip, x);
          loaded = true;
        }
      }
      if (!loaded) {
#pragma unroll
        for (int i = 0; i < DIN; ++i) x[i] = ip[i * n0];
      }
      line_apply<T, DIN, DOUT, SYM>(E, x, y);
    } else {
      constexpr int NA = NIN + (EX ? 1 : 0);
      T x[NA][DIN];
#pragma unroll
      for (int a = 0; a < NA; ++a) {
        const T* p = EX && a == NIN ? extra + ib : ip + (size_t)a * ks;
#pragma unroll
        for (int i = 0; i < DIN; ++i) x[a][i] = p[i * n0];
      }
      line_apply_sum<T, NA, DIN, DOUT, SYM>(E, x, y);
    }
    if constexpr (VOUT) {
      if (n0 == 1 && (reinterpret_cast<uintptr_t>(op) & 15) == 0) {
        vec_store<T, DOUT>(op, y);
        continue;
      }
    }
#pragma unroll
    for (int q = 0; q < DOUT; ++q) op[q * n0] = y[q];
  }
}
// FP64: one function per shape, not inlined (the code of an integer line is long; the axes share it)
template <int DIN, int DOUT, int SYM, int NIN, bool EX, int OG, int IBS, int OBS>
__device__ __noinline__ void lines_fp64(const double* in, int ks, const double* extra, double* out, EoFp64 E, int nlines,
                                        int n0, uint32_t magic) {
  lines_body<double, DIN, DOUT, SYM, NIN, EX, OG, IBS, OBS>(in, ks, extra, out, E, nlines, n0, magic, threadIdx.x,
                                                            blockDim.x);
}
template <typename T, int N0, int DIN, int DOUT, int SYM, int NIN = 1, bool EX = false, int OG = 0, int IBS = 0,
          int OBS = 0>
__device__ __forceinline__ void lines(const T* in, T* out, Eo<T> E, int nouter, int ks = 0, const T* extra = nullptr) {
  constexpr uint32_t magic = N0 > 1 ? (uint32_t)((0x100000000ull + N0 - 1) / N0) : 0u;  // l / N0 for l N0 < 2^32
  if constexpr (sizeof(T) == 8)
    lines_fp64<DIN, DOUT, SYM, NIN, EX, OG, IBS, OBS>(in, ks, extra, out, E, nouter * N0, N0, magic);
  else
    lines_body<T, DIN, DOUT, SYM, NIN, EX, OG, IBS, OBS>(in, ks, extra, out, E, nouter * N0, N0, magic, threadIdx.x,
                                                         blockDim.x);
}

// V_d <- D~_d V_d + the shares of the two faces of direction d, in place.  V: [nb][5][N^3]; F: the cells' face
// shares [nb][6][2][5][N^2] (global).  The line's operator takes D_0, L_0, the N values, -L_1, D_1: with the sign
// of L_1 it is antisymmetric under reflection like D~ itself.
template <typename T, int N, int D>
__device__ __forceinline__ void lift_body(T* V, const T* __restrict__ F, Eo<T> E, int nb, bool vol) {
  constexpr int N2 = N * N, N3 = N2 * N, st = D == 0 ? 1 : (D == 1 ? N : N2);
  for (int l = threadIdx.x; l < nb * 5 * N2; l += blockDim.x) {
    const int ec = l / N2, j = l - ec * N2, e = ec / 5, c = ec - 5 * e;
    const T* f0 = F + (size_t)e * fbuf_per_cell<N>() + (2 * D * 2 * 5 + c) * N2 + j;
    const T* f1 = f0 + 2 * 5 * N2;
    T x[N + 4], y[N];
    x[0] = f0[5 * N2];
    x[1] = f0[0];
    x[N + 2] = -f1[0];
    x[N + 3] = f1[5 * N2];
    T* v = V + ec * N3 + face_node<N>(D, 0, j % N, j / N);
#pragma unroll
    for (int i = 0; i < N; ++i) x[2 + i] = vol ? v[i * st] : T(0);
    line_apply<T, N + 4, N, -1>(E, x, y);
#pragma unroll
    for (int i = 0; i < N; ++i) v[i * st] = y[i];
  }
}
template <int N>
__device__ __noinline__ void lift_fp64(double* V, const double* F, EoFp64 E, int nb, bool vol, int n3) {
  // the three directions one after the other, V_d n3 values apart
  lift_body<double, N, 0>(V, F, E, nb, vol);
  lift_body<double, N, 1>(V + n3, F, E, nb, vol);
  lift_body<double, N, 2>(V + 2 * n3, F, E, nb, vol);
}

// ---------------------------------------------------------------------------
// Point fluxes
// ---------------------------------------------------------------------------
// Convective flux through a face with unit normal n (any normal, or n = sgn e_D when AFF), LLF:
// f = ({{F_c}} + lambda/2 [[U]]) . n.  Components in physical order.
template <typename T, int D, bool AFF>
__device__ __forceinline__ void llf_side(const T u[5], const T n[3], T sgn, const PhysT<T>& ph, T f[5], T& lam) {
  const T rinv = rcp_of(ph.rho_r + u[0]);
  const T m2 = u[1] * u[1] + u[2] * u[2] + u[3] * u[3];
  const T dp = ph.gm1 * (u[4] - T(0.5) * rinv * m2);
  lam = sqrt_of(m2) * rinv + sqrt_of(fabs(ph.gamma * (ph.p_r + dp) * rinv));
  const T mn = AFF ? sgn * u[1 + D] : u[1] * n[0] + u[2] * n[1] + u[3] * n[2];
  const T vn = mn * rinv;
  f[0] = mn;
  f[1] = u[1] * vn;
  f[2] = u[2] * vn;
  f[3] = u[3] * vn;
  if (AFF) {
    f[1 + D] += sgn * dp;
  } else {
    f[1] += dp * n[0];
    f[2] += dp * n[1];
    f[3] += dp * n[2];
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
// tangential ones, those of rho, m_D and the tangential momentum along its own direction enter.
// gd: normal derivatives (physical order); r1, d1, a1: d/dx_t1 of rho, m_D, m_t1; r2, d2, a2: d/dx_t2 of
// rho, m_D, m_t2.  f: components (m_D, m_t1, m_t2, rho E).
template <typename T, int D>
__device__ __forceinline__ void visc_normal(const SideState<T>& s, const T gd[5], T r1, T d1, T a1, T r2, T d2, T a2,
                                            const PhysT<T>& ph, T f[4]) {
  constexpr int t1 = D == 0 ? 1 : 0, t2 = D == 2 ? 1 : 2;
  const T ad = (gd[1 + D] - s.v[D] * gd[0]) * s.rinv;
  const T at1 = (gd[1 + t1] - s.v[t1] * gd[0]) * s.rinv;
  const T at2 = (gd[1 + t2] - s.v[t2] * gd[0]) * s.rinv;
  const T b1 = (d1 - s.v[D] * r1) * s.rinv;
  const T b2 = (d2 - s.v[D] * r2) * s.rinv;
  const T cc = ((a1 - s.v[t1] * r1) + (a2 - s.v[t2] * r2)) * s.rinv;
  f[0] = ph.mu * (T(4) / T(3) * ad - T(2) / T(3) * cc);
  f[1] = ph.mu * (at1 + b1);
  f[2] = ph.mu * (at2 + b2);
  const T q = (gd[4] - s.E * gd[0]) * s.rinv - (s.v[D] * ad + s.v[t1] * at1 + s.v[t2] * at2);
  f[3] = f[0] * s.v[D] + f[1] * s.v[t1] + f[2] * s.v[t2] + ph.lam_cv * q;
}

// F_v(U, j (x) e_D) on an axis-aligned face: normal column fd (m_D, m_t1, m_t2, rho E) and the nonzero entries
// (m_D, m_t, rho E) of the tangential columns.
template <typename T, int D>
__device__ __forceinline__ void visc_jump(const SideState<T>& s, const T j[5], const PhysT<T>& ph, T fd[4], T f1[3],
                                          T f2[3]) {
  constexpr int t1 = D == 0 ? 1 : 0, t2 = D == 2 ? 1 : 2;
  const T mr = ph.mu * s.rinv;
  const T gd = mr * (j[1 + D] - s.v[D] * j[0]);
  const T g1 = mr * (j[1 + t1] - s.v[t1] * j[0]);
  const T g2 = mr * (j[1 + t2] - s.v[t2] * j[0]);
  const T h = T(-2) / T(3) * gd;
  fd[0] = T(4) / T(3) * gd;
  fd[1] = g1;
  fd[2] = g2;
  // lambda/c_v ((j_E - E j_0)/rho - v . g/mu), g/mu = (j_m - v j_0)/rho
  const T v2 = s.v[0] * s.v[0] + s.v[1] * s.v[1] + s.v[2] * s.v[2];
  const T q = j[4] - s.E * j[0] - (s.v[0] * j[1] + s.v[1] * j[2] + s.v[2] * j[3] - v2 * j[0]);
  fd[3] = fd[0] * s.v[D] + g1 * s.v[t1] + g2 * s.v[t2] + (ph.lam_cv * s.rinv) * q;
  f1[0] = g1;
  f1[1] = h;
  f1[2] = g1 * s.v[D] + h * s.v[t1];
  f2[0] = g2;
  f2[1] = h;
  f2[2] = g2 * s.v[D] + h * s.v[t2];
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
#pragma unroll
  for (int i = 0; i < 3; ++i) r.g[i] = mr * (j[1 + i] - s.v[i] * j[0]);
  r.h = T(-2) / T(3) * (r.g[0] * n[0] + r.g[1] * n[1] + r.g[2] * n[2]);
  const T v2 = s.v[0] * s.v[0] + s.v[1] * s.v[1] + s.v[2] * s.v[2];
  r.q = (ph.lam_cv * s.rinv) *
        (j[4] - s.E * j[0] - (s.v[0] * j[1] + s.v[1] * j[2] + s.v[2] * j[3] - v2 * j[0]));
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
template <int N, int QC>
struct CollSizes {
  static constexpr int N2 = N * N, N3 = N2 * N, PC = QC * QC * QC;
  static constexpr int F = PC > N3 ? PC : N3;
  static constexpr int PER_CELL = 15 * F + 20 * N3;
};
template <typename T, int N, int QC, int QV, int CB>
constexpr size_t coll_cell_smem() {
  return ((size_t)table_elems<T, N, QC, QV>() + (size_t)CB * CollSizes<N, QC>::PER_CELL) * sizeof(T) + 64;
}

// Cells per CTA and threads.
template <typename T, int N, int QC, int QV>
constexpr int coll_cells() {
  int cb = 2;
  while (cb > 1 && ((size_t)table_elems<T, N, QC, QV>() + (size_t)cb * CollSizes<N, QC>::PER_CELL) * sizeof(T) > 74 * 1024)
    --cb;
  return cb;
}
// Threads: 128, and more where only two (FP64) or four (FP32) large cells fit an SM.  Measured: FP64 k = 3, 2 cells
// and 128 threads 14.9 ms per stage at 64^3 (192 threads 17.4, one cell 17.9 to 23.6); FP64 k = 5, 40^3, 192 threads
// 15.2 ms (128: 18.5, 256: 27.0, their registers no longer hold the point fluxes); FP32 k = 5, 256 threads 1.30 ms
// (128: 1.67, 192: 1.34); FP32 k = 3 stored, 32^3, 2 cells and 128 threads 0.264 ms (256: 0.326; one cell 0.277).
template <typename T, int N, int QC, int QV>
constexpr int coll_threads() {
  constexpr size_t smem = coll_cell_smem<T, N, QC, QV, coll_cells<T, N, QC, QV>()>();
  return sizeof(T) == 8 ? (smem > 64 * 1024 ? 192 : 128) : (smem > 40 * 1024 ? 256 : 128);
}
template <typename T, int N, int QC, int QV>
constexpr int coll_ctas() {  // resident CTAs that the registers have to allow
  const int b = (int)(227 * 1024 / coll_cell_smem<T, N, QC, QV, coll_cells<T, N, QC, QV>()>());
  return b < 1 ? 1 : (b > 4 ? 4 : b);
}

// kp.out_mode: 0 writes F(U), 1 L(U), 2 the stage update (as dg_op_kernel).
template <typename T, int N, int QC, int QV, int CB, int GEO>
__global__ void __launch_bounds__(coll_threads<T, N, QC, QV>(), coll_ctas<T, N, QC, QV>())
    dg_coll_cell_kernel(const KParams kp, const double* __restrict__ U,
                                                                         T* Rout, T* dU, double* Uout) {
  static_assert(QV == N && GEO != GEO_FLY, "collocation form");
  using S = CollSizes<N, QC>;
  constexpr int N2 = S::N2, N3 = S::N3, PC = S::PC, NTH = coll_threads<T, N, QC, QV>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* stab = reinterpret_cast<T*>(smem_raw);
  T* F0 = stab + table_elems<T, N, QC, QV>();
  T* F1 = F0 + CB * 5 * S::F;
  T* F2 = F1 + CB * 5 * S::F;
  T* V = F2 + CB * 5 * S::F;  // [3][CB][5][N^3]
  T* Ug = V + 3 * CB * 5 * N3;
  constexpr int VS = CB * 5 * N3;
  const int e0 = blockIdx.x * CB;
  const int nb = min(CB, kp.Nc - e0);
  const Tab<T> tb = load_tables<T, N, QC, QV>(static_cast<const T*>(kp.tables), stab);
  const PhysT<T> ph = make_phys<T>(kp);
  const KConst<T>& kc = kconst<T>(kp);
  const size_t base = (size_t)e0 * 5 * N3;
  const int nvals = nb * 5 * N3, nbl = nb * 5;
  constexpr int PER = (CB * 5 * N3 + NTH - 1) / NTH;
  const T* Ud = static_cast<const T*>(kp.Udev);
  if (Ud)
    batched_pass<PER>(threadIdx.x, NTH, nvals, [&](int i) { return Ud[base + i]; }, [&](int i, T v) { F0[i] = v; });
  else
    batched_pass<PER>(threadIdx.x, NTH, nvals, [&](int i) { return U[base + i]; }, [&](int i, double v) {
      F0[i] = dev_value<T>(kp, v, (i / N3) % 5);
    });
  __syncthreads();
  const bool conv = kp.conv != 0, visc = kp.visc != 0;
  const bool force = kp.has_bf && kp.out_mode != 0;
  // 1-3. values at the convective and at the viscous points
  if (conv) lines<T, 1, N, QC, 1>(F0, F1, tb.eSc, nbl * N2);
  lines<T, 1, N, N, 1>(F0, V, tb.eSm, nbl * N2);
  __syncthreads();
  if (conv) lines<T, QC, N, QC, 1>(F1, F2, tb.eSc, nbl * N);
  lines<T, N, N, N, 1>(V, V + VS, tb.eSm, nbl * N);
  __syncthreads();
  if (conv) lines<T, QC * QC, N, QC, 1>(F2, F0, tb.eSc, nbl);
  lines<T, N2, N, N, 1>(V + VS, Ug, tb.eSm, nbl);
  __syncthreads();
  // 4. convective flux (point arithmetic); reference gradients at the viscous points (sweeps)
  if (conv) {
    for (int idx = threadIdx.x; idx < nb * PC; idx += NTH) {
      const int e = idx / PC, p = idx - e * PC, o = e * 5 * PC + p;
      T u[5];
#pragma unroll
      for (int c = 0; c < 5; ++c) u[c] = F0[o + c * PC];
      const T rinv = rcp_of(ph.rho_r + u[0]);
      const T dp = pressure_dev(u, rinv, ph.gm1);
      const T Hr = (ph.H_r + u[4] + dp) * rinv;
      T* Fd[3] = {F0, F1, F2};
      if (GEO == GEO_AFFINE) {
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const T m = kc.hinv[j] * u[1 + j];
          const T a = m * rinv;
          T* f = Fd[j] + o;
          f[0] = m;
#pragma unroll
          for (int i = 0; i < 3; ++i) f[(1 + i) * PC] = i == j ? u[1 + i] * a + kc.hinv[j] * dp : u[1 + i] * a;
          f[4 * PC] = Hr * m;
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
          f[0] = m;
          f[PC] = m * v[0] + dp * j0;
          f[2 * PC] = m * v[1] + dp * j1;
          f[3 * PC] = m * v[2] + dp * j2;
          f[4 * PC] = Hr * m;
        }
      }
    }
  }
  if (visc) {
    lines<T, 1, N, N, -1>(Ug, V, tb.eDv, nbl * N2);
    lines<T, N, N, N, -1>(Ug, V + VS, tb.eDv, nbl * N);
    lines<T, N2, N, N, -1>(Ug, V + 2 * VS, tb.eDv, nbl);
  }
  __syncthreads();
  // 5. viscous flux with the sign of -F (point arithmetic); D~ of the convective flux, in place (sweeps)
  if (visc) {
    for (int idx = threadIdx.x; idx < nb * N3; idx += NTH) {
      const int e = idx / N3, p = idx - e * N3, o = e * 5 * N3 + p;
      T u[5], G[5][3];
      T* v0 = V + o;
#pragma unroll
      for (int c = 0; c < 5; ++c) u[c] = Ug[o + c * N3];
      T Jd[9];
      if (GEO == GEO_AFFINE) {
#pragma unroll
        for (int c = 0; c < 5; ++c)
#pragma unroll
          for (int j = 0; j < 3; ++j) G[c][j] = kc.hinv[j] * v0[j * VS + c * N3];
      } else {
        const T* g = static_cast<const T*>(kp.gcv) + (size_t)(e0 + e) * 10 * N3 + p;
#pragma unroll
        for (int m = 0; m < 9; ++m) Jd[m] = g[m * N3];
#pragma unroll
        for (int c = 0; c < 5; ++c) {
          const T g0 = v0[c * N3], g1 = v0[VS + c * N3], g2 = v0[2 * VS + c * N3];
#pragma unroll
          for (int a = 0; a < 3; ++a) G[c][a] = Jd[a] * g0 + Jd[3 + a] * g1 + Jd[6 + a] * g2;
        }
        const T dj = -g[9 * N3];
#pragma unroll
        for (int m = 0; m < 9; ++m) Jd[m] *= dj;
      }
      const SideState<T> s = side_state(u, ph);
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
        f[0] = T(0);
        if (GEO == GEO_AFFINE) {
          const T w = -kc.hinv[b];
#pragma unroll
          for (int i = 0; i < 3; ++i) f[(1 + i) * N3] = w * t[i][b];
          f[4 * N3] = w * q[b];
        } else {
          const T j0 = Jd[3 * b], j1 = Jd[3 * b + 1], j2 = Jd[3 * b + 2];
#pragma unroll
          for (int i = 0; i < 3; ++i) f[(1 + i) * N3] = j0 * t[i][0] + j1 * t[i][1] + j2 * t[i][2];
          f[4 * N3] = j0 * q[0] + j1 * q[1] + j2 * q[2];
        }
      }
    }
  }
  if (conv) {
    lines<T, 1, QC, QC, -1>(F0, F0, tb.eDcW, nbl * QC * QC);
    lines<T, QC, QC, QC, -1>(F1, F1, tb.eDcW, nbl * QC);
    lines<T, QC * QC, QC, QC, -1>(F2, F2, tb.eDcW, nbl);
  }
  __syncthreads();
  // 6-8. projection of the summed convective parts onto the l_g; D~ and face shares of the viscous arrays
  const T* FBc = static_cast<const T*>(kp.fbuf) + (size_t)e0 * fbuf_per_cell<N>();
  if (conv) lines<T, QC * QC, QC, N, 1, 3, false, 0, 0, PC>(F0, F0, tb.ePc, nbl, CB * 5 * S::F);
  if constexpr (sizeof(T) == 8) {
    lift_fp64<N>(V, FBc, tb.eLift, nb, visc, VS);
  } else {
    lift_body<T, N, 0>(V, FBc, tb.eLift, nb, visc);
    lift_body<T, N, 1>(V + VS, FBc, tb.eLift, nb, visc);
    lift_body<T, N, 2>(V + 2 * VS, FBc, tb.eLift, nb, visc);
  }
  __syncthreads();
  if (conv) {
    lines<T, QC, QC, N, 1, 1, false, N, PC>(F0, F1, tb.ePc, nbl * N);
    __syncthreads();
    lines<T, 1, QC, N, 1>(F1, F2, tb.ePc, nbl * N2);
  } else {
    for (int i = threadIdx.x; i < nvals; i += NTH) F2[i] = T(0);
  }
  __syncthreads();
  // 9-11. M^-1 in the l_g basis is a scaling by 1/|J| (affine: in the flux scales); S^-1 back to the nodes
  T* sr = F2;
  if (GEO == GEO_AFFINE && !force && kp.out_mode != 0) {
    lines<T, 1, N, N, 1, 3, true>(V, F1, tb.eSmi, nbl * N2, VS, F2);
  } else {
    for (int i = threadIdx.x; i < nvals; i += NTH) {
      const int p = i % N3, e = i / (5 * N3), c = (i / N3) % 5;
      T r = F2[i] + (V[i] + (V[VS + i] + V[2 * VS + i]));
      if (kp.out_mode == 0) {
        const T w = tb.wm[p % N] * tb.wm[(p / N) % N] * tb.wm[p / N2];
        r *= GEO == GEO_AFFINE ? -w * kc.detJ : -w;
      } else {
        if (GEO == GEO_STORED) r *= rcp_of(static_cast<const T*>(kp.gm)[(size_t)(e0 + e) * N3 + p]);
        if (force && c > 0) {
          const T* ug = Ug + e * 5 * N3 + p;
          r += c < 4 ? kc.bf[c - 1]
                     : (kc.bf[0] * ug[N3] + kc.bf[1] * ug[2 * N3] + kc.bf[2] * ug[3 * N3]) * rcp_of(ph.rho_r + ug[0]);
        }
      }
      F0[i] = r;
    }
    __syncthreads();
    lines<T, 1, N, N, 1>(F0, F1, kp.out_mode == 0 ? tb.eSvT : tb.eSmi, nbl * N2);
  }
  __syncthreads();
  lines<T, N, N, N, 1>(F1, F0, kp.out_mode == 0 ? tb.eSvT : tb.eSmi, nbl * N);
  __syncthreads();
  lines<T, N2, N, N, 1>(F0, sr, kp.out_mode == 0 ? tb.eSvT : tb.eSmi, nbl);
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
template <typename T, int N, int QC, int QV, int FB_>
constexpr size_t coll_face_smem() {
  return ((size_t)table_elems<T, N, QC, QV>() + (size_t)FB_ * (CollFaceSizes<N, QC>::PER_FACE + 1)) * sizeof(T) +
         3 * FB_ * sizeof(int) + 64;
}
template <typename T, int N, int QC, int QV>
constexpr int coll_faces() {
  int fb = 8;
  while (fb > 1 && ((size_t)table_elems<T, N, QC, QV>() + (size_t)fb * CollFaceSizes<N, QC>::PER_FACE) * sizeof(T) > 56 * 1024)
    --fb;
  return fb;
}
template <typename T>
constexpr int coll_face_threads() {
  return 128;
}

template <typename T, int N, int QC, int QV, int FB_, int D, int GEO>
__device__ __forceinline__ void coll_face_terms(const double* __restrict__ U, const T* __restrict__ Ud, const int* eo,
                                                const int* en, const int* oc, const T* tau_f, T* sm, const Tab<T>& tb,
                                                const KParams& kp, const PhysT<T>& ph, int nb, int s, T* __restrict__ FBuf) {
  using Z = CollFaceSizes<N, QC>;
  constexpr int N2 = N * N, N3 = N2 * N, QC2 = QC * QC, NTH = coll_face_threads<T>();
  constexpr int t1 = D == 0 ? 1 : 0, t2 = D == 2 ? 1 : 2;
  constexpr bool AFF = GEO == GEO_AFFINE;
  const KConst<T>& kc = kconst<T>(kp);
  const int f = 2 * D + s, fo = 2 * D + (1 - s);
  const T sgn = s ? T(1) : T(-1);
  const int idm = s ? N - 1 : 0, idp = s ? 0 : N - 1;
  const T* dlm = s ? tb.dl1 : tb.dl0;
  const T* dlp = s ? tb.dl0 : tb.dl1;
  const int nf = nb * N2, nl = 5 * nf;  // values per slot and per array
  T* VV = sm;                      // [Lm, Lp, Dm, Dp][5][nb][N2]
  T* TT = VV + FB_ * Z::VV;        // [t1 m, t1 p, t2 m, t2 p][5 (3 used if AFF)][nb][N2]
  T* C0 = TT + FB_ * Z::TT;
  T* C1 = C0 + FB_ * Z::C0;        // [m, p][5][nb][QC2]; later the convective share [5][nb][N2]
  const bool conv = kp.conv != 0, visc = kp.visc != 0;
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
    T dm = T(0), dp = T(0), vm = T(0), vp = T(0);
#pragma unroll
    for (int i = 0; i < N; ++i) {
      dm += dlm[i] * a[i];
      dp += dlp[i] * b[i];
      if (i == idm) vm = a[i];
      if (i == idp) vp = b[i];
    }
    VV[idx] = vm;
    VV[nl + idx] = vp;
    VV[2 * nl + idx] = dm;
    VV[3 * nl + idx] = dp;
  }
  __syncthreads();
  if (conv) lines<T, 1, N, QC, 1>(VV, C0, tb.eSc, 2 * 5 * nb * N);
  if (visc) lines<T, 1, N, N, 1>(VV, TT, tb.eSm, 4 * 5 * nb * N);
  __syncthreads();
  if (conv) lines<T, QC, N, QC, 1>(C0, C1, tb.eSc, 2 * 5 * nb);
  if (visc) lines<T, N, N, N, 1>(TT, VV, tb.eSm, 4 * 5 * nb);
  __syncthreads();
  // convective flux (point arithmetic); tangential derivatives (sweeps)
  if (conv) {
    const int nc = nb * QC2;
    for (int idx = threadIdx.x; idx < nc; idx += NTH) {
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
      llf_side<T, D, AFF>(um, n, sgn, ph, fm, lm);
      llf_side<T, D, AFF>(up, n, sgn, ph, fp, lp);
      const T lam = lm > lp ? lm : lp;
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        const int c = slot_comp<D>(q);
        C1[q * nc + idx] = w * (fm[c] + fp[c] + lam * (um[c] - up[c]));
      }
    }
  }
  if (visc) {
    if (AFF) {
#pragma unroll
      for (int sd = 0; sd < 2; ++sd) {
        lines<T, 1, N, N, -1>(VV + sd * nl, TT + sd * nl, tb.eDv, 3 * nb * N);
        lines<T, N, N, N, -1>(VV + sd * nl + nf, TT + (2 + sd) * nl, tb.eDv, 3 * nb);
      }
    } else {
      lines<T, 1, N, N, -1>(VV, TT, tb.eDv, 2 * 5 * nb * N);
      lines<T, N, N, N, -1>(VV, TT + 2 * nl, tb.eDv, 2 * 5 * nb);
    }
  }
  __syncthreads();
  // viscous fluxes (point arithmetic); projection of the convective flux (sweeps).  Shares are of -F.
  if (visc) {
    for (int idx = threadIdx.x; idx < nf; idx += NTH) {
      const int e = idx / N2, p = idx - e * N2;
      const bool wall = en[e] < 0;
      T um[5], up[5], jmp[5];
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        um[slot_comp<D>(q)] = VV[q * nf + idx];
        up[slot_comp<D>(q)] = VV[nl + q * nf + idx];
      }
      if (wall) wall_ghost(um, ph, up);
      const SideState<T> sm_ = side_state(um, ph), sp_ = side_state(up, ph);
      const T tau = tau_f[e];
#pragma unroll
      for (int c = 0; c < 5; ++c) jmp[c] = um[c] - up[c];
      T fm[4], fp[4];
      if (AFF) {
        const T hd = kc.hinv[D], h1 = kc.hinv[t1], h2 = kc.hinv[t2];
        T* T1m = TT + idx;
        T* T1p = T1m + nl;
        T* T2m = T1p + nl;
        T* T2p = T2m + nl;
        T gm[5], gp[5];
#pragma unroll
        for (int q = 0; q < 5; ++q) {
          gm[slot_comp<D>(q)] = hd * VV[2 * nl + q * nf + idx];
          gp[slot_comp<D>(q)] = hd * VV[3 * nl + q * nf + idx];
        }
        visc_normal<T, D>(sm_, gm, h1 * T1m[nf], h1 * T1m[2 * nf], h1 * T1m[0], h2 * T2m[0], h2 * T2m[nf],
                          h2 * T2m[2 * nf], ph, fm);
        if (wall) {
          // grad U+ = grad U-, at the ghost state
          visc_normal<T, D>(sp_, gm, h1 * T1m[nf], h1 * T1m[2 * nf], h1 * T1m[0], h2 * T2m[0], h2 * T2m[nf],
                            h2 * T2m[2 * nf], ph, fp);
        } else {
          visc_normal<T, D>(sp_, gp, h1 * T1p[nf], h1 * T1p[2 * nf], h1 * T1p[0], h2 * T2p[0], h2 * T2p[nf],
                            h2 * T2p[2 * nf], ph, fp);
        }
        // value share (own side): (V, Q*.n), Q*.n = {{F_v}}.n - tau [[U]]; the other side's is the negative
        const T wv = T(0.5) * sgn * hd, wt = hd * tau;
        const int fs[5] = {1, -1, 0, 2, 3};  // slot -> entry of fm
#pragma unroll
        for (int q = 0; q < 5; ++q) {
          const T t = -wt * jmp[slot_comp<D>(q)];
          VV[q * nf + idx] = fs[q] < 0 ? t : t + wv * (fm[fs[q] < 0 ? 0 : fs[q]] + fp[fs[q] < 0 ? 0 : fs[q]]);
        }
        // +1/2 (grad V, F_v(U, [[U]])), [[U]] = sgn jmp (x) e_D
        const T hw = T(0.5) * sgn * hd;
        T a[4], b1[3], b2[3];
        visc_jump<T, D>(sm_, jmp, ph, a, b1, b2);
        VV[2 * nl + idx] = hw * hd * a[1];
        VV[2 * nl + nf + idx] = T(0);
        VV[2 * nl + 2 * nf + idx] = hw * hd * a[0];
        VV[2 * nl + 3 * nf + idx] = hw * hd * a[2];
        VV[2 * nl + 4 * nf + idx] = hw * hd * a[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          T1m[i * nf] = hw * h1 * b1[i];
          T2m[i * nf] = hw * h2 * b2[i];
        }
        if (!wall) visc_jump<T, D>(sp_, jmp, ph, a, b1, b2);
        VV[3 * nl + idx] = hw * hd * a[1];
        VV[3 * nl + nf + idx] = T(0);
        VV[3 * nl + 2 * nf + idx] = hw * hd * a[0];
        VV[3 * nl + 3 * nf + idx] = hw * hd * a[2];
        VV[3 * nl + 4 * nf + idx] = hw * hd * a[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          T1p[i * nf] = hw * h1 * b1[i];
          T2p[i * nf] = hw * h2 * b2[i];
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
              dst[b][q * nf] = c == 0 ? T(0) : r[c == 0 ? 0 : c - 1];
            }
          }
        }
      }
    }
  }
  if (conv) lines<T, QC, QC, N, 1>(C1, C0, tb.ePc, 5 * nb);
  __syncthreads();
  // tangential gradient tests, in place; the convective share
  if (visc) {
    if (AFF) {
#pragma unroll
      for (int sd = 0; sd < 2; ++sd) {
        lines<T, 1, N, N, -1>(TT + sd * nl, TT + sd * nl, tb.eDvW, 3 * nb * N);
        lines<T, N, N, N, -1>(TT + (2 + sd) * nl, TT + (2 + sd) * nl, tb.eDvW, 3 * nb);
      }
    } else {
      lines<T, 1, N, N, -1>(TT, TT, tb.eDvW, 2 * 5 * nb * N);
      lines<T, N, N, N, -1>(TT + 2 * nl, TT + 2 * nl, tb.eDvW, 2 * 5 * nb);
    }
  }
  if (conv) lines<T, 1, QC, N, 1>(C0, C1, tb.ePc, 5 * nb * N);
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
      if (AFF) {
        // tested entries: along t1 (m_D, m_t1, rho E), along t2 (m_D, m_t2, rho E)
        const int k1 = sl == 2 ? 0 : (sl == 0 ? 1 : (sl == 4 ? 2 : -1));
        const int k2 = sl == 2 ? 0 : (sl == 3 ? 1 : (sl == 4 ? 2 : -1));
        if (k1 >= 0) {
          lm += TT[k1 * nf + r];
          lp += TT[nl + k1 * nf + r];
        }
        if (k2 >= 0) {
          lm += TT[2 * nl + k2 * nf + r];
          lp += TT[3 * nl + k2 * nf + r];
        }
      } else {
        lm += TT[idx] + TT[2 * nl + idx];
        lp += TT[nl + idx] + TT[3 * nl + idx];
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
__global__ void __launch_bounds__(coll_face_threads<T>()) dg_coll_face_kernel(const KParams kp,
                                                                              const double* __restrict__ U,
                                                                              T* __restrict__ FBuf) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* stab = reinterpret_cast<T*>(smem_raw);
  T* sm = stab + table_elems<T, N, QC, QV>();
  T* tau_f = sm + FB_ * CollFaceSizes<N, QC>::PER_FACE;
  int* eo = reinterpret_cast<int*>(tau_f + FB_);
  int* en = eo + FB_;
  int* oc = en + FB_;
  const int d = blockIdx.y;
  int s, nb;
  if (!face_batch<FB_>(kp, d, s, nb, eo, en, oc, tau_f)) return;
  const Tab<T> tb = load_tables<T, N, QC, QV>(static_cast<const T*>(kp.tables), stab);
  const PhysT<T> ph = make_phys<T>(kp);
  __syncthreads();
  const T* Ud = static_cast<const T*>(kp.Udev);
  const int* ocp = kp.flist ? oc : nullptr;
  if (d == 0)
    coll_face_terms<T, N, QC, QV, FB_, 0, GEO>(U, Ud, eo, en, ocp, tau_f, sm, tb, kp, ph, nb, s, FBuf);
  else if (d == 1)
    coll_face_terms<T, N, QC, QV, FB_, 1, GEO>(U, Ud, eo, en, ocp, tau_f, sm, tb, kp, ph, nb, s, FBuf);
  else
    coll_face_terms<T, N, QC, QV, FB_, 2, GEO>(U, Ud, eo, en, ocp, tau_f, sm, tb, kp, ph, nb, s, FBuf);
}

// Where the collocation kernels are used.
template <typename T, int N, int QC, int QV, int GEO>
constexpr bool coll_ok() {
  return QV == N && coll_rule(N, QV) && GEO != GEO_FLY && coll_cell_smem<T, N, QC, QV, 1>() <= 227 * 1024;
}

template <typename T, int N, int QC, int QV, int GEO>
int launch_coll_cell(const KParams& kp, const double* U, void* Rout, void* dU, double* Uout, cudaStream_t st) {
  constexpr int CB = coll_cells<T, N, QC, QV>();
  constexpr size_t smem = coll_cell_smem<T, N, QC, QV, CB>();
  static_assert(smem <= 227 * 1024, "cell kernel shared memory");
  auto k = dg_coll_cell_kernel<T, N, QC, QV, CB, GEO>;
  static bool attr[kMaxDevices] = {};
  if (smem_attr_once(k, smem, attr)) return -1;
  k<<<(kp.Nc + CB - 1) / CB, coll_threads<T, N, QC, QV>(), smem, st>>>(kp, U, static_cast<T*>(Rout), static_cast<T*>(dU), Uout);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

template <typename T, int N, int QC, int QV, int GEO>
int launch_coll_faces(const KParams& kp, const double* U, void* FB, cudaStream_t st) {
  constexpr int FB_ = coll_faces<T, N, QC, QV>();
  constexpr size_t smem = coll_face_smem<T, N, QC, QV, FB_>();
  static_assert(smem <= 227 * 1024, "face kernel shared memory");
  auto k = dg_coll_face_kernel<T, N, QC, QV, FB_, GEO>;
  static bool attr[kMaxDevices] = {};
  if (smem_attr_once(k, smem, attr)) return -1;
  k<<<dim3(face_blocks(kp, FB_), 3), coll_face_threads<T>(), smem, st>>>(kp, U, static_cast<T*>(FB));
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace dgcns
