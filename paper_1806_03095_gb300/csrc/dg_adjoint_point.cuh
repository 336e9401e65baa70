// Transposed pointwise Jacobians (vector-Jacobian products) of the flux
// routines of dg_kernels.cuh, hand-derived in reverse order of the forward
// statements.  Every function ACCUMULATES into its adjoint outputs.
#pragma once
#include "dg_kernels.cuh"

namespace dgcns {

// ub += (dF_c/du)^T Fb for the convective flux in all three directions,
// Fb[a][c] = adjoint of F_c[c][a] (deviation form: pressure deviation dp).
template <typename T>
__device__ __forceinline__ void conv_flux_vjp(const T u[5], const T Fb[3][5], const PhysT<T>& ph, T ub[5]) {
  const T rinv = rcp_of(ph.rho_r + u[0]);
  const T m[3] = {u[1], u[2], u[3]};
  const T v[3] = {m[0] * rinv, m[1] * rinv, m[2] * rinv};
  const T msq = m[0] * m[0] + m[1] * m[1] + m[2] * m[2];
  const T dp = ph.gm1 * (u[4] - T(0.5) * rinv * msq);
  T vb[3] = {T(0), T(0), T(0)}, mb[3] = {T(0), T(0), T(0)};
  T dpb = T(0), u4b = T(0), rinvb = T(0);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    mb[a] += Fb[a][0];  // F[0][a] = m_a
#pragma unroll
    for (int i = 0; i < 3; ++i) {  // F[1+i][a] = m_i v_a + dp delta_ia
      mb[i] += Fb[a][1 + i] * v[a];
      vb[a] += Fb[a][1 + i] * m[i];
    }
    dpb += Fb[a][1 + a];
    // F[4][a] = (H_r + rhoE' + dp) v_a
    u4b += Fb[a][4] * v[a];
    dpb += Fb[a][4] * v[a];
    vb[a] += Fb[a][4] * (ph.H_r + u[4] + dp);
  }
  // dp = (gamma-1)(rhoE' - |m|^2 rinv / 2)
  u4b += ph.gm1 * dpb;
#pragma unroll
  for (int i = 0; i < 3; ++i) mb[i] -= ph.gm1 * rinv * m[i] * dpb;
  rinvb -= T(0.5) * ph.gm1 * msq * dpb;
  // v = m rinv
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    mb[i] += vb[i] * rinv;
    rinvb += vb[i] * m[i];
  }
  ub[0] -= rinv * rinv * rinvb;
  ub[1] += mb[0];
  ub[2] += mb[1];
  ub[3] += mb[2];
  ub[4] += u4b;
}

// ub += (dF_v/du)^T Fb, Gb += (dF_v/dG)^T Fb for F_v(u, G) (Fb[c][a], Gb[c][a]).
// With A_ij = Fb[1+i][j] + Fb[4][j] v_i (adjoint of tau), k_j = lambda/c_v Fb[4][j]:
//   adjoint of grad u:  gub_ij = mu (A_ij + A_ji) - 2/3 mu tr(A) delta_ij - k_j v_i,
// and D_ij = G[1+i][j] - v_i G[0][j] = gu_ij / rinv serves the stress, the heat flux and the adjoint of 1/rho.
template <typename T>
__device__ __forceinline__ void visc_flux_vjp(const T u[5], const T G[5][3], const T Fb[5][3], const PhysT<T>& ph,
                                              T ub[5], T Gb[5][3]) {
  const T rinv = rcp_of(ph.rho_r + u[0]);
  const T v[3] = {u[1] * rinv, u[2] * rinv, u[3] * rinv};
  const T E = (ph.rhoE_r + u[4]) * rinv;
  const T mr = ph.mu * rinv;
  T D[3][3], A[3][3], k[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    k[j] = ph.lam_cv * Fb[4][j];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      D[i][j] = G[1 + i][j] - v[i] * G[0][j];
      A[i][j] = Fb[1 + i][j] + Fb[4][j] * v[i];
    }
  }
  const T trD = T(2) / T(3) * (D[0][0] + D[1][1] + D[2][2]), trA = T(2) / T(3) * (A[0][0] + A[1][1] + A[2][2]);
  T vb[3] = {T(0), T(0), T(0)}, rinvb = T(0), Eb = T(0);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    T g0 = k[j] * E;  // -rho adjoint of G[0][j]
    const T e = mr * Fb[4][j], q = k[j] * rinv;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const T S = D[i][j] + D[j][i] - (i == j ? trD : T(0));
      const T gub = ph.mu * (A[i][j] + A[j][i] - (i == j ? trA : T(0))) - k[j] * v[i];
      vb[i] += e * S - q * D[i][j] - gub * (G[0][j] * rinv);
      Gb[1 + i][j] += gub * rinv;
      g0 += gub * v[i];
      rinvb += gub * D[i][j];
    }
    Gb[4][j] += q;
    Gb[0][j] -= g0 * rinv;
    Eb -= q * G[0][j];
    rinvb += k[j] * (G[4][j] - E * G[0][j]);
  }
  // E = (rhoE_r + rhoE') rinv, v = m rinv
  ub[4] += Eb * rinv;
  T t = Eb * E;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    ub[1 + i] += vb[i] * rinv;
    t += vb[i] * v[i];
  }
  ub[0] -= rinv * (rinv * rinvb + t);
}

// The two viscous transposes of a face, for any unit normal n, or e_DIR when AFF (the sign of the normal is then in the
// weights): only the entries of the normal column, row and diagonal enter.
//
// Normal flux F_v(u, G) n with the adjoint b of its components: A = a n^T, a_i = b_{1+i} + b_4 v_i, so
// gub_ij = p_i n_j + n_i s_j - h delta_ij with k = lambda/c_v b_4, s = mu a, p = s - k v, h = 2/3 s.n.
template <typename T, int DIR, bool AFF>
__device__ __forceinline__ void visc_normal_vjp(const T u[5], const T G[5][3], const T n[3], const T b[5],
                                                const PhysT<T>& ph, T ub[5], T Gb[5][3]) {
  const T rinv = rcp_of(ph.rho_r + u[0]);
  const T v[3] = {u[1] * rinv, u[2] * rinv, u[3] * rinv};
  const T E = (ph.rhoE_r + u[4]) * rinv;
  const T mr = ph.mu * rinv, k = ph.lam_cv * b[4];
  auto dot = [&](T x, T y, T z) { return AFF ? (DIR == 0 ? x : (DIR == 1 ? y : z)) : x * n[0] + y * n[1] + z * n[2]; };
  T D[3][3], p[3], s[3], Dn[3], nD[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    s[i] = ph.mu * (b[1 + i] + b[4] * v[i]);
    p[i] = s[i] - k * v[i];
#pragma unroll
    for (int j = 0; j < 3; ++j)
      D[i][j] = AFF && i != DIR && j != DIR && i != j ? T(0) : G[1 + i][j] - v[i] * G[0][j];
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    Dn[i] = dot(D[i][0], D[i][1], D[i][2]);
    nD[i] = dot(D[0][i], D[1][i], D[2][i]);
  }
  const T h = T(2) / T(3) * dot(s[0], s[1], s[2]), trD = D[0][0] + D[1][1] + D[2][2];
  const T nG0 = dot(G[0][0], G[0][1], G[0][2]), nG4 = dot(G[4][0], G[4][1], G[4][2]);
  const T nv = dot(v[0], v[1], v[2]), pv = p[0] * v[0] + p[1] * v[1] + p[2] * v[2];
  const T sG = s[0] * G[0][0] + s[1] * G[0][1] + s[2] * G[0][2];
  // adjoint of 1/rho in gu = D rinv and gE = (G4 - E G0) rinv
  const T rinvb = p[0] * Dn[0] + p[1] * Dn[1] + p[2] * Dn[2] + (s[0] * nD[0] + s[1] * nD[1] + s[2] * nD[2]) - h * trD +
                  k * (nG4 - E * nG0);
  const T kr = k * rinv, b4 = mr * b[4], nc = pv + k * E;
  T t = T(0);
  T vb[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const T ni = AFF ? (i == DIR ? T(1) : T(0)) : n[i];
    // v in tau n . v, in the heat flux and in D
    const T tn = AFF ? (i == DIR ? T(2) * Dn[i] - T(2) / T(3) * trD : Dn[i] + nD[i]) : Dn[i] + nD[i] - T(2) / T(3) * trD * ni;
    const T w = AFF ? (i == DIR ? p[i] * nG0 + sG - h * G[0][i] : p[i] * nG0 - h * G[0][i])
                    : p[i] * nG0 + ni * sG - h * G[0][i];
    vb[i] = b4 * tn - kr * Dn[i] - rinv * w;
    t += vb[i] * v[i];
    ub[1 + i] += vb[i] * rinv;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      if (AFF && i != DIR && j != DIR && i != j) continue;
      T g;
      if (AFF)
        g = (j == DIR ? p[i] : T(0)) + (i == DIR ? s[j] : T(0)) - (i == j ? h : T(0));
      else
        g = p[i] * n[j] + n[i] * s[j] - (i == j ? h : T(0));
      Gb[1 + i][j] += g * rinv;
    }
    const T nj = ni;  // column i of the rho and energy rows
    if (AFF) {
      Gb[0][i] -= rinv * ((i == DIR ? nc : T(0)) + nv * s[i] - h * v[i]);
      if (i == DIR) Gb[4][i] += kr;
    } else {
      Gb[0][i] -= rinv * (nc * nj + nv * s[i] - h * v[i]);
      Gb[4][i] += kr * nj;
    }
  }
  const T Eb = -kr * nG0;
  ub[4] += Eb * rinv;
  ub[0] -= rinv * (rinv * rinvb + t + Eb * E);
}

// Jump flux F_v(u, j (x) n) with the adjoint Fb of its entries: gu = g n^T, g = (j_m - v j_0) rinv;
// A = Fb_m + v Fb_E^T, gb = mu (A n + A^T n - 2/3 tr(A) n) - k v, k = lambda/c_v Fb_E . n.  jb += adjoint of j.
template <typename T, int DIR, bool AFF>
__device__ __forceinline__ void visc_jump_vjp(const T u[5], const T j[5], const T n[3], const T Fb[5][3],
                                              const PhysT<T>& ph, T ub[5], T jb[5]) {
  const T rinv = rcp_of(ph.rho_r + u[0]);
  const T v[3] = {u[1] * rinv, u[2] * rinv, u[3] * rinv};
  const T E = (ph.rhoE_r + u[4]) * rinv;
  auto dot = [&](T x, T y, T z) { return AFF ? (DIR == 0 ? x : (DIR == 1 ? y : z)) : x * n[0] + y * n[1] + z * n[2]; };
  T A[3][3], d[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    d[i] = j[1 + i] - v[i] * j[0];  // g / rinv
#pragma unroll
    for (int a = 0; a < 3; ++a) A[i][a] = AFF && i != DIR && a != DIR && i != a ? T(0) : Fb[1 + i][a] + Fb[4][a] * v[i];
  }
  const T trA = T(2) / T(3) * (A[0][0] + A[1][1] + A[2][2]);
  const T en = dot(Fb[4][0], Fb[4][1], Fb[4][2]), k = ph.lam_cv * en;
  const T dn = dot(d[0], d[1], d[2]), de = d[0] * Fb[4][0] + d[1] * Fb[4][1] + d[2] * Fb[4][2];
  const T mr = ph.mu * rinv, kr = k * rinv;
  const T j0r = j[0] * rinv, h = T(2) / T(3) * dn;
  T rinvb = k * (j[4] - E * j[0]), gv = T(0), t = T(0);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const T An = dot(A[i][0], A[i][1], A[i][2]), nA = dot(A[0][i], A[1][i], A[2][i]);
    T q, te;  // mu-free parts of gb_i and of (tau e)_i / rinv
    if (AFF) {
      q = i == DIR ? T(2) * An - trA : An + nA;
      te = i == DIR ? d[i] * en + de - h * Fb[4][i] : d[i] * en - h * Fb[4][i];
    } else {
      q = An + nA - trA * n[i];
      te = d[i] * en + n[i] * de - h * Fb[4][i];
    }
    const T gb = ph.mu * q - k * v[i];
    const T vb = mr * te - kr * d[i] - gb * j0r;
    jb[1 + i] += gb * rinv;
    gv += gb * v[i];
    rinvb += gb * d[i];
    ub[1 + i] += vb * rinv;
    t += vb * v[i];
  }
  jb[4] += kr;
  jb[0] -= rinv * (gv + k * E);
  const T Eb = -k * j0r;
  ub[4] += Eb * rinv;
  ub[0] -= rinv * (rinv * rinvb + t + Eb * E);
}

// ub += lb d(lambda)/du, lambda = |m|/rho + sqrt(|gamma p / rho|)
template <typename T>
__device__ __forceinline__ void wave_speed_vjp(const T u[5], T lb, const PhysT<T>& ph, T ub[5]) {
  const T rinv = T(1) / (ph.rho_r + u[0]);
  const T msq = u[1] * u[1] + u[2] * u[2] + u[3] * u[3];
  const T mn = sqrt(msq);
  const T dp = ph.gm1 * (u[4] - T(0.5) * rinv * msq);
  const T P = ph.p_r + dp;
  const T s = ph.gamma * P * rinv;
  const T c = sqrt(fabs(s));
  T rinvb = lb * mn;
  if (mn > T(0)) {
#pragma unroll
    for (int i = 0; i < 3; ++i) ub[1 + i] += lb * rinv * u[1 + i] / mn;
  }
  if (c > T(0)) {
    const T sb = lb * (s >= T(0) ? T(1) : T(-1)) / (T(2) * c);
    const T Pb = sb * ph.gamma * rinv;
    rinvb += sb * ph.gamma * P;
    ub[4] += ph.gm1 * Pb;
#pragma unroll
    for (int i = 0; i < 3; ++i) ub[1 + i] -= ph.gm1 * rinv * u[1 + i] * Pb;
    rinvb -= T(0.5) * ph.gm1 * msq * Pb;
  }
  ub[0] -= rinv * rinv * rinvb;
}

template <typename T>
__device__ __forceinline__ T wave_speed(const T u[5], const PhysT<T>& ph) {
  const T rinv = T(1) / (ph.rho_r + u[0]);
  const T msq = u[1] * u[1] + u[2] * u[2] + u[3] * u[3];
  const T dp = ph.gm1 * (u[4] - T(0.5) * rinv * msq);
  return sqrt(msq) * rinv + sqrt(fabs(ph.gamma * (ph.p_r + dp) * rinv));
}

// umb += (d ghost / d um)^T upb for the wall state of wall_ghost().
template <typename T>
__device__ __forceinline__ void wall_ghost_vjp(const T um[5], const T upb[5], const PhysT<T>& ph, T umb[5]) {
  const T rinv = T(1) / (ph.rho_r + um[0]);
  const T msq = um[1] * um[1] + um[2] * um[2] + um[3] * um[3];
  // up4 = cvTw2 um0 - um4 + |m|^2 rinv
  umb[0] += upb[0] + upb[4] * (ph.cvTw2 - msq * rinv * rinv);
#pragma unroll
  for (int i = 0; i < 3; ++i) umb[1 + i] += -upb[1 + i] + upb[4] * T(2) * um[1 + i] * rinv;
  umb[4] -= upb[4];
}

// Local Lax--Friedrichs face point: flux[c] = w (1/2 sum_a (F(um)+F(up))[c][a] n_a + Lambda/2 (um-up)_c)
// with Lambda = max(lambda(um), lambda(up)).  Given fb = adjoint of flux.
template <typename T>
__device__ __forceinline__ void llf_vjp(const T um[5], const T up[5], const T n[3], T w, const T fb[5],
                                        const PhysT<T>& ph, T umb[5], T upb[5]) {
  T Fb[3][5];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int c = 0; c < 5; ++c) Fb[a][c] = T(0.5) * w * fb[c] * n[a];
  conv_flux_vjp(um, Fb, ph, umb);
  conv_flux_vjp(up, Fb, ph, upb);
  const T lm = wave_speed(um, ph), lp = wave_speed(up, ph);
  const T lam = lm > lp ? lm : lp;  // same branch as the forward flux (ties: the up side)
  T lamb = T(0);
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    umb[c] += T(0.5) * w * lam * fb[c];
    upb[c] -= T(0.5) * w * lam * fb[c];
    lamb += T(0.5) * w * fb[c] * (um[c] - up[c]);
  }
  if (lm > lp)
    wave_speed_vjp(um, lamb, ph, umb);
  else
    wave_speed_vjp(up, lamb, ph, upb);
}

// The same for the face-centric kernels: the normal flux F_c n transposed as such (b = w/2 fb; n any unit normal or
// e_DIR when AFF, ws then carries its sign), the wave speed of the faster side only.
template <typename T, int DIR, bool AFF>
__device__ __forceinline__ void conv_normal_vjp(const T u[5], const T n[3], const T b[5], const PhysT<T>& ph, T rinv, T dp,
                                                T ub[5]) {
  auto dot = [&](T x, T y, T z) { return AFF ? (DIR == 0 ? x : (DIR == 1 ? y : z)) : x * n[0] + y * n[1] + z * n[2]; };
  const T mn = dot(u[1], u[2], u[3]), vn = mn * rinv;
  const T msq = u[1] * u[1] + u[2] * u[2] + u[3] * u[3];
  // f = (mn, m vn + dp n, (H_r + rhoE' + dp) vn), vn = mn rinv
  const T vnb = b[1] * u[1] + b[2] * u[2] + b[3] * u[3] + b[4] * (ph.H_r + u[4] + dp);
  const T dpb = dot(b[1], b[2], b[3]) + b[4] * vn;
  const T mnb = b[0] + vnb * rinv, c = ph.gm1 * rinv * dpb;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    T t = b[1 + i] * vn - c * u[1 + i];
    if (AFF) {
      if (i == DIR) t += mnb;
    } else {
      t += mnb * n[i];
    }
    ub[1 + i] += t;
  }
  ub[4] += b[4] * vn + ph.gm1 * dpb;
  ub[0] -= rinv * rinv * (vnb * mn - ph.hgm1 * msq * dpb);
}
template <typename T, int DIR, bool AFF>
__device__ __forceinline__ void llf_pair_vjp(const T um[5], const T up[5], const T n[3], T w, T ws, const T fb[5],
                                             const PhysT<T>& ph, T umb[5], T upb[5]) {
  T b[5];
#pragma unroll
  for (int c = 0; c < 5; ++c) b[c] = T(0.5) * ws * fb[c];
  const T rm = rcp_of(ph.rho_r + um[0]), rp = rcp_of(ph.rho_r + up[0]);
  const T dm = pressure_dev(um, rm, ph.gm1), dpp = pressure_dev(up, rp, ph.gm1);
  conv_normal_vjp<T, DIR, AFF>(um, n, b, ph, rm, dm, umb);
  conv_normal_vjp<T, DIR, AFF>(up, n, b, ph, rp, dpp, upb);
  const T qm = um[1] * um[1] + um[2] * um[2] + um[3] * um[3], qp = up[1] * up[1] + up[2] * up[2] + up[3] * up[3];
  const T am = sqrt_of(qm), ap = sqrt_of(qp);
  const T sm = ph.gamma * (ph.p_r + dm) * rm, sp = ph.gamma * (ph.p_r + dpp) * rp;
  const T cm = sqrt_of(fabs(sm)), cp = sqrt_of(fabs(sp));
  const T lm = am * rm + cm, lp = ap * rp + cp;
  const bool own = lm > lp;  // same branch as the forward flux (ties: the up side)
  const T hl = T(0.5) * w * (own ? lm : lp);
  T lb = T(0);
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    umb[c] += hl * fb[c];
    upb[c] -= hl * fb[c];
    lb += fb[c] * (um[c] - up[c]);
  }
  lb *= T(0.5) * w;
  // the faster side's lambda = a rinv + c, c = sqrt(|s|), s = gamma p rinv
  const T a = own ? am : ap, r = own ? rm : rp, c = own ? cm : cp, s = own ? sm : sp, msq = own ? qm : qp;
  T rinvb = lb * a, kv = a > T(0) ? lb * r * rcp_of(a) : T(0), eb = T(0);
  if (c > T(0)) {
    const T sb = lb * T(0.5) * rcp_of(c) * (s >= T(0) ? T(1) : T(-1));
    const T Pb = sb * ph.gamma * r;
    rinvb += sb * ph.gamma * (own ? ph.p_r + dm : ph.p_r + dpp) - ph.hgm1 * msq * Pb;
    eb = ph.gm1 * Pb;
    kv -= eb * r;
  }
  const T r0 = r * r * rinvb;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const T x = kv * (own ? um[1 + i] : up[1 + i]);
    if (own)
      umb[1 + i] += x;
    else
      upb[1 + i] += x;
  }
  if (own) {
    umb[0] -= r0;
    umb[4] += eb;
  } else {
    upb[0] -= r0;
    upb[4] += eb;
  }
}

// Viscous face point of one side's face term (own side "m"):
//   val[c] = -w (1/2 sum_a (F_v(um,Gm) + F_v(up,Gp))[c][a] n_a - tau (um - up)_c)   tested with V
//   Ft_b[c] = -1/2 w sum_a Jm[b][a] F_v(um, (um - up) (x) n)[c][a]                 tested with d_b V
// Given yv (adjoint of val) and yb[b] (adjoint of Ft_b), accumulate umb, Gmb, upb, Gpb (physical gradients).
template <typename T>
__device__ __forceinline__ void sipg_vjp(const T um[5], const T Gm[5][3], const T up[5], const T Gp[5][3],
                                         const T n[3], const T Jm[9], T w, T tau, const T yv[5], const T yb[3][5],
                                         const PhysT<T>& ph, T umb[5], T Gmb[5][3], T upb[5], T Gpb[5][3]) {
  T jmp[5], jmpb[5];
  T Jg[5][3], Jgb[5][3], Fb[5][3];
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    jmp[c] = um[c] - up[c];
    jmpb[c] = w * tau * yv[c];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      Jg[c][a] = jmp[c] * n[a];
      Jgb[c][a] = T(0);
      Fb[c][a] = T(-0.5) * w * (Jm[a] * yb[0][c] + Jm[3 + a] * yb[1][c] + Jm[6 + a] * yb[2][c]);
    }
  }
  visc_flux_vjp(um, Jg, Fb, ph, umb, Jgb);
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    jmpb[c] += Jgb[c][0] * n[0] + Jgb[c][1] * n[1] + Jgb[c][2] * n[2];
#pragma unroll
    for (int a = 0; a < 3; ++a) Fb[c][a] = T(-0.5) * w * yv[c] * n[a];
  }
  visc_flux_vjp(um, Gm, Fb, ph, umb, Gmb);
  visc_flux_vjp(up, Gp, Fb, ph, upb, Gpb);
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    umb[c] += jmpb[c];
    upb[c] -= jmpb[c];
  }
}

}  // namespace dgcns
