// Face-centric face kernel of the mixed form (FP32 arithmetic), affine meshes: the same face terms as
// face_pair_terms (Sec. 2.2.2: LLF flux, SIPG flux and the -1/2 (grad V, F_v(U, [[U]])) term; both cells'
// shares of every face once), organised so that every 1D contraction runs in registers:
//
//  1. trace tasks, one thread per (face, side, component): the thread reads its cell's component block as
//     x-lines, forms the face-layer values L and the normal derivatives D at the face nodes, interpolates
//     L to the convective and viscous face points, differentiates along both tangents by collocation and
//     interpolates D; the 2D tensor contractions of a face are held in the thread's registers, and each
//     result goes to shared memory once;
//  2. convective points, one thread per (face, point): the LLF flux, tested with the own side's V (the
//     other side's test is its negative); viscous points, one thread per (face, point): the SIPG flux and
//     F_v(U^-+, [[U]] (x) n) of both sides;
//  3. test tasks, one thread per (face, side, component): the transposed contractions in registers, and the
//     two shares (value and normal derivative) written to the face buffer.
//
// Point fluxes, signs and the face buffer are those of the collocation form (dg_coll.cuh): no quadrature
// weights, and a viscous integrand at the face's Gauss points is a share as it stands.  The even-odd 1D
// operators come from constant memory with compile-time offsets.  k = 3, TGV 64^3, per launch:
// 1.42 -> 1.14 ms against the form that tested with the nodal basis and formed all flux columns.
#pragma once
#include "dg_coll.cuh"

namespace dgcns {

// One 1D line through an even-odd operator (DOUT x DIN, symmetry SYM) in registers: y = O x.
template <int DIN, int DOUT, int SYM>
__device__ __forceinline__ void eo_apply(const float* __restrict__ E, const float (&x)[DIN], float (&y)[DOUT]) {
  constexpr int IH = DIN / 2, OH = (DOUT + 1) / 2;
  const float* A = E;
  const float* B = E + OH * IH;
  const float* C = E + 2 * OH * IH;
  float xe[IH > 0 ? IH : 1], xo[IH > 0 ? IH : 1];
#pragma unroll
  for (int i = 0; i < IH; ++i) {
    xe[i] = x[i] + x[DIN - 1 - i];
    xo[i] = x[i] - x[DIN - 1 - i];
  }
#pragma unroll
  for (int q = 0; q < OH; ++q) {
    float e = (DIN & 1) ? C[q] * x[IH] : 0.f;
    float o = 0.f;
#pragma unroll
    for (int i = 0; i < IH; ++i) {
      e = fmaf(A[q * IH + i], xe[i], e);
      o = fmaf(B[q * IH + i], xo[i], o);
    }
    y[q] = e + o;
    if (!((DOUT & 1) && q == OH - 1)) y[DOUT - 1 - q] = SYM > 0 ? e - o : o - e;
  }
}

// K consecutive floats between registers and memory: 16-byte vectors when K is a multiple of 4 (the
// address then 16-byte aligned), else scalars.
template <int K>
__device__ __forceinline__ void arr_load(const float* p, float (&x)[K]) {
  if constexpr (K % 4 == 0) {
    vec_load<float, K>(p, x);
  } else {
#pragma unroll
    for (int i = 0; i < K; ++i) x[i] = p[i];
  }
}

template <int K>
__device__ __forceinline__ void arr_store(float* p, const float (&x)[K]) {
  if constexpr (K % 4 == 0) {
    vec_store<float, K>(p, x);
  } else {
#pragma unroll
    for (int i = 0; i < K; ++i) p[i] = x[i];
  }
}

// 2D tensor contraction in registers: X[NI1][NI0] (index 0 fastest) -> Y[NO1][NO0] with operator E0 along
// index 0 and E1 along index 1 (either may be the identity: NI == NO and E == nullptr is not used; every
// call applies both).
template <int NI0, int NI1, int NO0, int NO1, int SYM0, int SYM1>
__device__ __forceinline__ void eo_2d(const float* __restrict__ E0, const float* __restrict__ E1,
                                      const float (&X)[NI1 * NI0], float (&Y)[NO1 * NO0]) {
  float T[NI1][NO0];
#pragma unroll
  for (int b = 0; b < NI1; ++b) {
    float x[NI0], y[NO0];
#pragma unroll
    for (int a = 0; a < NI0; ++a) x[a] = X[b * NI0 + a];
    eo_apply<NI0, NO0, SYM0>(E0, x, y);
#pragma unroll
    for (int a = 0; a < NO0; ++a) T[b][a] = y[a];
  }
#pragma unroll
  for (int a = 0; a < NO0; ++a) {
    float x[NI1], y[NO1];
#pragma unroll
    for (int b = 0; b < NI1; ++b) x[b] = T[b][a];
    eo_apply<NI1, NO1, SYM1>(E1, x, y);
#pragma unroll
    for (int b = 0; b < NO1; ++b) Y[b * NO0 + a] = y[b];
  }
}

// Contraction along index 0 only: X[NB][NI] -> Y[NB][NO].
template <int NI, int NO, int NB, int SYM>
__device__ __forceinline__ void eo_dir0(const float* __restrict__ E, const float (&X)[NB * NI], float (&Y)[NB * NO]) {
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    float x[NI], y[NO];
#pragma unroll
    for (int a = 0; a < NI; ++a) x[a] = X[b * NI + a];
    eo_apply<NI, NO, SYM>(E, x, y);
#pragma unroll
    for (int a = 0; a < NO; ++a) Y[b * NO + a] = y[a];
  }
}

// Contraction along index 1 only: X[NI][NA] -> Y[NO][NA].
template <int NI, int NO, int NA, int SYM>
__device__ __forceinline__ void eo_dir1(const float* __restrict__ E, const float (&X)[NI * NA], float (&Y)[NO * NA]) {
#pragma unroll
  for (int a = 0; a < NA; ++a) {
    float x[NI], y[NO];
#pragma unroll
    for (int b = 0; b < NI; ++b) x[b] = X[b * NA + a];
    eo_apply<NI, NO, SYM>(E, x, y);
#pragma unroll
    for (int b = 0; b < NO; ++b) Y[b * NA + a] = y[b];
  }
}

// Face-layer values L and normal derivatives D (sum_i dl_i u_i along the normal lines) at the face nodes
// (j1 along the first tangent, fastest) of one component block src [N^3] of a cell, the face at layer
// id (0 or N-1) along direction DIR; the block is read as its N^2 x-lines.
template <int N, int DIR>
__device__ __forceinline__ void face_traces(const float* src, const float* __restrict__ dl, int id,
                                            float (&L)[N * N], float (&D)[N * N]) {
  const bool last = id != 0;
#pragma unroll
  for (int j = 0; j < N * N; ++j) D[j] = 0.f;
#pragma unroll
  for (int zz = 0; zz < N; ++zz)
#pragma unroll
    for (int yy = 0; yy < N; ++yy) {
      float x[N];
      if constexpr ((N * sizeof(float)) % 16 == 0) {
        vec_load<float, N>(src + (zz * N + yy) * N, x);
      } else {
#pragma unroll
        for (int a = 0; a < N; ++a) x[a] = src[(zz * N + yy) * N + a];
      }
      if constexpr (DIR == 0) {  // face node (y, z), layer x
        const int j = yy + N * zz;
        float acc = 0.f;
#pragma unroll
        for (int a = 0; a < N; ++a) acc = fmaf(dl[a], x[a], acc);
        D[j] = acc;
        L[j] = last ? x[N - 1] : x[0];
      } else if constexpr (DIR == 1) {  // face node (x, z), layer y
        const float w = dl[yy];
#pragma unroll
        for (int a = 0; a < N; ++a) D[a + N * zz] = fmaf(w, x[a], D[a + N * zz]);
        if (yy == 0 && !last) {
#pragma unroll
          for (int a = 0; a < N; ++a) L[a + N * zz] = x[a];
        }
        if (yy == N - 1 && last) {
#pragma unroll
          for (int a = 0; a < N; ++a) L[a + N * zz] = x[a];
        }
      } else {  // face node (x, y), layer z
        const float w = dl[zz];
#pragma unroll
        for (int a = 0; a < N; ++a) D[a + N * yy] = fmaf(w, x[a], D[a + N * yy]);
        if (zz == 0 && !last) {
#pragma unroll
          for (int a = 0; a < N; ++a) L[a + N * yy] = x[a];
        }
        if (zz == N - 1 && last) {
#pragma unroll
          for (int a = 0; a < N; ++a) L[a + N * yy] = x[a];
        }
      }
    }
}

// Shared-memory layout of one CTA (floats): per face, conv traces [2][5][QC^2] (the own side's slots
// later hold the LLF integrand), viscous traces [2][5][VS] with VS >= 4 QV^2 (U, d/dt1, d/dt2, normal
// derivative; later the four test integrands).  Padding against shared-memory bank conflicts: a (side, component) task writes and reads its 4 QV^2 viscous values as
// 16-byte vectors, so VS = 4 QV^2 + 4 puts the blocks of 8 neighbouring tasks on distinct banks (a stride
// of 4 QV^2 = 64 words put them all on the same 4 banks); the per-face stride is 8 (mod 32) words, so the
// tasks of the next face in the same quarter-warp land on other banks too.
template <int N, int QC, int QV>
struct TaskFaceSizes {
  static constexpr int PC = QC * QC, PV = QV * QV;
  static constexpr int CIN = (2 * 5 * PC + 3) & ~3;
  static constexpr int VS = 4 * PV + 4;
  static constexpr int VIN = 2 * 5 * VS;
  static constexpr int RAW = CIN + VIN;
  static constexpr int PER_FACE = RAW + ((8 - RAW % 32) + 32) % 32;
};

template <int N, int QC, int QV, int FPB>
constexpr size_t task_face_smem_bytes() {
  return ((size_t)table_elems<float, N, QC, QV>() + (size_t)FPB * TaskFaceSizes<N, QC, QV>::PER_FACE + 3 * FPB) *
             sizeof(float) + 64;
}

// Phases 1-4 of the task kernel for faces normal to direction DIR (compile-time, so that the small
// per-point arrays indexed by direction stay in registers).
template <int N, int QC, int QV, int FPB, int NTH, int DIR>
__device__ __forceinline__ void face_task_body(const KParams& kp, float* FB, const Tab<float>& tb,
                                               const PhysT<float>& ph, float* sface, const float* stau, const int* eo,
                                               const int* en, int nb, int s) {
  using S = TaskFaceSizes<N, QC, QV>;
  constexpr int N2 = N * N, N3 = N * N * N, PC = S::PC, PV = S::PV;
  constexpr int d = DIR, t1 = DIR == 0 ? 1 : 0, t2 = DIR == 2 ? 1 : 2;
  const KConst<float>& kc = kconst<float>(kp);
  const float hinv_d = kc.hinv[d];
  const float sgn = s ? 1.f : -1.f;
  const float* Ud = static_cast<const float*>(kp.Udev);

  // 1. trace tasks (face b, side sd: 0 own / 1 other, component c)
  for (int task = threadIdx.x; task < nb * 10; task += NTH) {
    const int b = task / 10, r = task - 10 * b, sd = r / 5, c = r - 5 * sd;
    const int cell = sd ? en[b] : eo[b];
    if (cell < 0) continue;  // wall: the ghost state is formed at the points
    const int id = (sd ? 1 - s : s) ? N - 1 : 0;  // the face's layer index along d in this cell
    const float* dl = (sd ? 1 - s : s) ? tb.dl1 : tb.dl0;
    const float* src = Ud + ((size_t)cell * 5 + c) * N3;
    float L[N2], D[N2];
    face_traces<N, DIR>(src, dl, id, L, D);
    float* fb = sface + b * S::PER_FACE;
    if (kp.conv) {
      float Uc[PC];
      eo_2d<N, N, QC, QC, 1, 1>(tb.eSc, tb.eSc, L, Uc);
      float* o = fb + (sd * 5 + c) * PC;
#pragma unroll
      for (int p = 0; p < PC; ++p) o[p] = Uc[p];
    }
    if (kp.visc) {
      float Uv[PV], G[PV];
      float* o = fb + S::CIN + (sd * 5 + c) * S::VS;
      eo_2d<N, N, QV, QV, 1, 1>(tb.eSv, tb.eSv, L, Uv);
      arr_store<PV>(o, Uv);
      eo_dir0<QV, QV, QV, -1>(tb.eDv, Uv, G);
      arr_store<PV>(o + PV, G);
      eo_dir1<QV, QV, QV, -1>(tb.eDv, Uv, G);
      arr_store<PV>(o + 2 * PV, G);
      eo_2d<N, N, QV, QV, 1, 1>(tb.eSv, tb.eSv, D, G);
      arr_store<PV>(o + 3 * PV, G);
    }
  }
  __syncthreads();

  // 2. convective points: LLF integrand of the own side (the other side's is its negative)
  if (kp.conv) {
    // one face per warp and pass: the points of two faces on one warp would share banks
    static_assert(PC <= 32, "points of a face in one warp");
    for (int b = threadIdx.x / 32; b < nb; b += NTH / 32) {
      const int p = threadIdx.x % 32;
      if (p >= PC) continue;
      float* fb = sface + b * S::PER_FACE;
      float um[5], up[5];
#pragma unroll
      for (int c = 0; c < 5; ++c) um[c] = fb[c * PC + p];
      if (en[b] < 0) {
        wall_ghost(um, ph, up);
      } else {
#pragma unroll
        for (int c = 0; c < 5; ++c) up[c] = fb[(5 + c) * PC + p];
      }
      const float nd[3] = {0.f, 0.f, 0.f};
      float fm[5], fp[5], lm, lp;
      const float w = -0.5f * hinv_d;
      llf_side<float, DIR, true>(um, nd, sgn * w, ph, fm, lm);
      llf_side<float, DIR, true>(up, nd, sgn * w, ph, fp, lp);
      const float lam = w * (lm > lp ? lm : lp);
#pragma unroll
      for (int c = 0; c < 5; ++c) fb[c * PC + p] = fm[c] + fp[c] + lam * (um[c] - up[c]);
    }
  }

  // viscous points: value share (V, Q*.n) and the +1/2 (grad V, F_v(U, [[U]] (x) n)) integrands of both sides
  if (kp.visc) {
    // two faces per warp, b and b + 2: their blocks start 16 banks apart (neighbours only 8)
    for (int task = threadIdx.x; task < ((nb + 3) & ~3) * PV; task += NTH) {
      const int bt = task / PV, p = task - PV * bt, b = (bt & ~3) | (bt & 1) << 1 | (bt >> 1 & 1);
      if (b >= nb) continue;
      const bool wall = en[b] < 0;
      float* vm = sface + b * S::PER_FACE + S::CIN + p;
      float* vp = vm + 5 * S::VS;
      float um[5], up[5], jmp[5], gd[5], fm[4], fp[4];
#pragma unroll
      for (int c = 0; c < 5; ++c) um[c] = vm[c * S::VS];
      if (wall) {
        wall_ghost(um, ph, up);
      } else {
#pragma unroll
        for (int c = 0; c < 5; ++c) up[c] = vp[c * S::VS];
      }
      const SideState<float> sm = side_state(um, ph), sp = side_state(up, ph);
      auto normal = [&](const SideState<float>& st, const float* v, float f[4]) {
        const float *g1 = v + PV, *g2 = v + 2 * PV;
#pragma unroll
        for (int c = 0; c < 5; ++c) gd[c] = v[c * S::VS + 3 * PV];
        visc_normal<float, DIR>(st, gd, g1[0], g1[(1 + d) * S::VS], g1[(1 + t1) * S::VS], g2[0], g2[(1 + d) * S::VS],
                                g2[(1 + t2) * S::VS], kc, f);
      };
      normal(sm, vm, fm);
      normal(sp, wall ? vm : vp, fp);  // wall: grad U+ = grad U-, at the ghost state
      const float wv = 0.5f * sgn * hinv_d, wt = hinv_d * stau[b];
      float v[5];
#pragma unroll
      for (int c = 0; c < 5; ++c) {
        jmp[c] = um[c] - up[c];
        v[c] = -wt * jmp[c];
      }
      v[1 + d] += wv * (fm[0] + fp[0]);
      v[1 + t1] += wv * (fm[1] + fp[1]);
      v[1 + t2] += wv * (fm[2] + fp[2]);
      v[4] += wv * (fm[3] + fp[3]);
      // [[U]] = sgn jmp (x) e_d
#pragma unroll
      for (int c = 0; c < 5; ++c) jmp[c] *= sgn;
      auto tests = [&](const SideState<float>& st, float* q, float sg) {
        float a[4], b1[3], b2[3];
        visc_jump<float, DIR>(st, jmp, kc, a, b1, b2);
#pragma unroll
        for (int c = 0; c < 5; ++c) q[c * S::VS] = sg * v[c];
        float* q1 = q + PV;
        q1[0] = q1[(1 + t2) * S::VS] = 0.f;
        q1[(1 + d) * S::VS] = b1[0];
        q1[(1 + t1) * S::VS] = b1[1];
        q1[4 * S::VS] = b1[2];
        float* q2 = q + 2 * PV;
        q2[0] = q2[(1 + t1) * S::VS] = 0.f;
        q2[(1 + d) * S::VS] = b2[0];
        q2[(1 + t2) * S::VS] = b2[1];
        q2[4 * S::VS] = b2[2];
        float* q3 = q + 3 * PV;
        q3[0] = 0.f;
        q3[(1 + d) * S::VS] = a[0];
        q3[(1 + t1) * S::VS] = a[1];
        q3[(1 + t2) * S::VS] = a[2];
        q3[4 * S::VS] = a[3];
      };
      tests(sm, vm, 1.f);
      if (!wall) tests(sp, vp, -1.f);
    }
  }
  __syncthreads();

  // 3. test tasks: value share L and normal-derivative share D of (face b, side sd, component c)
  for (int task = threadIdx.x; task < nb * 10; task += NTH) {
    const int b = task / 10, r = task - 10 * b, sd = r / 5, c = r - 5 * sd;
    const int cell = sd ? en[b] : eo[b];
    if (cell < 0) continue;
    const float* fb = sface + b * S::PER_FACE;
    float Ls[N2], Ds[N2];
#pragma unroll
    for (int j = 0; j < N2; ++j) {
      Ls[j] = 0.f;
      Ds[j] = 0.f;
    }
    if (kp.conv) {
      float X[PC], Y[N2];
      const float sg = sd ? -1.f : 1.f;
#pragma unroll
      for (int p = 0; p < PC; ++p) X[p] = sg * fb[c * PC + p];
      eo_2d<QC, QC, N, N, 1, 1>(tb.ePc, tb.ePc, X, Y);
#pragma unroll
      for (int j = 0; j < N2; ++j) Ls[j] = Y[j];
    }
    if (kp.visc) {
      const float* vi = fb + S::CIN + (sd * 5 + c) * S::VS;
      float G[PV], T[PV];
      arr_load<PV>(vi, G);
#pragma unroll
      for (int p = 0; p < PV; ++p) Ls[p] += G[p];
      arr_load<PV>(vi + PV, G);
      eo_dir0<QV, QV, QV, -1>(tb.eDvW, G, T);
#pragma unroll
      for (int p = 0; p < PV; ++p) Ls[p] += T[p];
      arr_load<PV>(vi + 2 * PV, G);
      eo_dir1<QV, QV, QV, -1>(tb.eDvW, G, T);
#pragma unroll
      for (int p = 0; p < PV; ++p) Ls[p] += T[p];
      arr_load<PV>(vi + 3 * PV, Ds);
    }
    const int f = 2 * d + (sd ? 1 - s : s);
    float* po = FB + (((size_t)cell * 6 + f) * 2 * 5 + c) * N2;
    arr_store<N2>(po, Ls);
    arr_store<N2>(po + 5 * N2, Ds);
  }
}

template <int N, int QC, int QV, int FPB, int NTH>
__global__ void __launch_bounds__(NTH) dg_face_task_kernel(const KParams kp, float* FB) {
  using S = TaskFaceSizes<N, QC, QV>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* stab = reinterpret_cast<float*>(smem_raw);
  float* sface = stab + ((table_elems<float, N, QC, QV>() + 3) & ~3);
  float* stau = sface + FPB * S::PER_FACE;
  int* eo = reinterpret_cast<int*>(stau + FPB);
  int* en = eo + FPB;
  const int d = blockIdx.y;
  int s, nb;
  const Tab<float> tb = load_tables<float, N, QC, QV>(static_cast<const float*>(kp.tables), stab);
  const PhysT<float> ph = make_phys<float>(kp);
  wait_for_predecessor();
  if (!face_batch<FPB>(kp, d, s, nb, eo, en, en, stau)) return;  // (no orientation codes: structured meshes only)
  __syncthreads();

  if (d == 0)
    face_task_body<N, QC, QV, FPB, NTH, 0>(kp, FB, tb, ph, sface, stau, eo, en, nb, s);
  else if (d == 1)
    face_task_body<N, QC, QV, FPB, NTH, 1>(kp, FB, tb, ph, sface, stau, eo, en, nb, s);
  else
    face_task_body<N, QC, QV, FPB, NTH, 2>(kp, FB, tb, ph, sface, stau, eo, en, nb, s);
}

// The task kernel serves the FP32 affine face terms at k = 3 (at k = 4 and 5 too few warps fit an SM: it was
// slower than the warp-per-face kernel there, measured).
template <int N, int QC, int QV>
constexpr bool task_faces_ok() {
  return N == 4 && coll_rule(N, QV);
}

template <int N, int QC, int QV, int FPB, int NTH>
int launch_task_faces_fpb(const KParams& kp, bool only_one_wave, void* FB, cudaStream_t st) {
  constexpr size_t smem = task_face_smem_bytes<N, QC, QV, FPB>();
  static_assert(smem <= 227 * 1024, "task face kernel shared memory");
  auto k = dg_face_task_kernel<N, QC, QV, FPB, NTH>;
  static bool attr[kMaxDevices] = {};
  static int per_sm[kMaxDevices] = {};
  if (smem_attr_once(k, smem, attr)) return -1;
  const int blocks = face_blocks(kp, FPB);
  if (only_one_wave && !one_wave(k, NTH, smem, 3ll * blocks, per_sm)) return 1;
  return launch_after(k, dim3(blocks, 3), NTH, smem, st, kp, static_cast<float*>(FB));
}
// 12 faces and 128 threads per CTA (120 trace and test tasks); on small meshes, as in dg_coll.cuh, 3 faces and one warp.
template <int N, int QC, int QV>
int launch_task_faces(const KParams& kp, void* FB, cudaStream_t st) {
  const int r = launch_task_faces_fpb<N, QC, QV, 3, 32>(kp, true, FB, st);
  return r <= 0 ? r : launch_task_faces_fpb<N, QC, QV, 12, 128>(kp, false, FB, st);
}

}  // namespace dgcns
