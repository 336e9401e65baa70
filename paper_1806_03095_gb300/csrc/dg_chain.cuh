// Chains of FP64 sweeps that stay in integers (dg_fixed.cuh) from one sweep to the next.
//
// A line that starts and ends in doubles spends more instructions on its conversions (about 16 per input and 24 per
// output) than on the contraction.  Inside a chain the values of a block (one component of one cell or of one face)
// stay integers relative to one exponent, that of the block's largest value: an operator of norm 2^n raises it by n
// at most, so every later exponent is known, nothing is normalised between sweeps, and in-place sums over the
// three directions are integer additions.  No exponent is shared by two cells or by two faces: a result depends on the
// cell and its neighbours only, not on what else its CTA carries (with one exponent per component of a CTA, a cell 2^-30
// of its batch neighbour lost 30 bits).
//
// Error: each sweep drops the bits below 2^-58 of the block's largest possible output; the bound grows by less than a
// bit per interpolation and by the norm per derivative.  Where sums cancel (the divergence of the fluxes, the
// total residual) the values fall far below that bound, so the next sweep first shifts each line up to the full
// width (RENORM) and ends in doubles, and a new chain starts from their maxima.  (Without this the error of L(U)
// at 40^3, k = 5 grew from 1.1e-14 to 5.5e-13.)  A chain ends with one rounding to 53 bits.
// A CTA that holds an exponent outside fx_exp_ok's range (NaN, infinities, denormals, extreme scales) takes the
// line-by-line sweeps for all its cells or faces, whose last bits may then differ.
#pragma once
#include "dg_kernels.cuh"

namespace dgcns {

// Exponent gain of one sweep that keeps `room` bits free above its outputs.
__device__ __forceinline__ int chain_gain(EoFp64 E, int room = 0) { return 64 - E.f[0].x - E.f[0].y + room; }

// Maxima of blocks: slot[q stride + i] takes the largest m[q] over the lanes of block i (0 where a lane has none).
// By atomics of the lanes, or, where blocks are runs of LEN > 16 consecutive lanes (the first and last may be shorter),
// one reduction per run and value; whole warps call.  Measured at 48^3, k = 3: cell kernel 4.0 ms (atomics of all lanes
// 4.5, reductions also for its runs of 16 4.05), face kernel 4.53 ms with atomics (reductions 4.86).
template <int LEN, int K>
__device__ __forceinline__ void block_max(uint32_t* slot, int stride, int i, const uint32_t (&m)[K]) {
  if constexpr (LEN <= 16) {
#pragma unroll
    for (int q = 0; q < K; ++q)
      if (m[q]) atomicMax(slot + q * stride + i, m[q]);
  } else {
    const int lane = threadIdx.x & 31, last = __shfl_sync(0xffffffffu, i, 31);
    for (int b = __shfl_sync(0xffffffffu, i, 0); b <= last; ++b) {
      uint32_t r = 0;
#pragma unroll
      for (int q = 0; q < K; ++q) {
        const uint32_t v = __reduce_max_sync(0xffffffffu, i == b ? m[q] : 0u);
        if (lane == q) r = v;
      }
      if (r) atomicMax(slot + lane * stride + b, r);
    }
  }
}
// All n blocks in the range of the chains (whole warps call).
__device__ __forceinline__ bool blocks_ok(const uint32_t* slot, int n) {
  bool ok = true;
  for (int i = threadIdx.x & 31; i < n; i += 32) ok = ok && fx_exp_ok(slot[i]);
  return __all_sync(0xffffffffu, ok);
}

enum { FROM_INT = 0, FROM_DOUBLE = 1, FROM_SUM = 2, TO_INT = 0, TO_DOUBLE = 1 };

// Shift a line up until its largest value has 61 bits; returns the shift.
template <int D>
__device__ __forceinline__ int fx_renorm(int64_t (&F)[D]) {
  uint64_t m = 0;
#pragma unroll
  for (int i = 0; i < D; ++i) m |= (uint64_t)(F[i] ^ (F[i] >> 63));
  const int s = max(__clzll((long long)m) - 3, 0) & 63;
#pragma unroll
  for (int i = 0; i < D; ++i) F[i] = (int64_t)((uint64_t)F[i] << s);
  return s;
}

// Lines as lines_fp64, in blocks of LPB lines (PER = LPB / n0 outer indices each).  A block's exponent is fx_exp(ex[b]) +
// add for integer inputs (value F 2^(exponent - 1083)) and without add for doubles; from block `nex` on the exponents
// repeat (a face's two sides).  Integer outputs keep `room` bits free.  FROM_SUM: the input is the sum of three integer
// arrays ks apart, renormalised, and the maxima of the outputs' blocks go to omax.
template <int DIN, int DOUT, int SYM, int IN, int OUT, int LPB, int PER, int OG, int IBS, int OBS>
__device__ __forceinline__ void chain_fp64(const double* in, int ks, double* out, EoFp64 E, int nlines, int n0,
                                        uint32_t magic, int nex, const uint32_t* ex, int add, int room, uint32_t* omax) {
  DGCNS_SHARED(in);
  DGCNS_SHARED(out);
  DGCNS_SHARED(E.f);
  DGCNS_SHARED(ex);
  const int t = E.f[0].x, sh = E.f[0].y - room;
  // (FROM_SUM: whole warps stay in the loop, for the reduction of the maxima)
#pragma unroll 1
  for (int l = threadIdx.x; (IN == FROM_SUM ? l & ~31 : l) < nlines; l += blockDim.x) {
    uint32_t m[1] = {0};
    if (IN != FROM_SUM || l < nlines) {
      const int outer = n0 > 1 ? (int)__umulhi((uint32_t)l, magic) : l;
      const int inner = l - outer * n0;
      const int ib = (OG > 0 ? (outer / (OG > 0 ? OG : 1)) * IBS + (outer % (OG > 0 ? OG : 1)) * n0 * DIN : outer * n0 * DIN) + inner;
      const int ob = (OBS > 0 ? outer * OBS : outer * n0 * DOUT) + inner;
      int64_t F[DIN], Y[DOUT];
      int e = 0;
      if (IN == FROM_DOUBLE || OUT == TO_DOUBLE) {
        const int b = outer / PER;
        e = fx_exp(ex[b < nex ? b : b - nex]);
      }
      if (IN == FROM_DOUBLE) {
        const double* ip = in + ib;
        double x[DIN];
#pragma unroll
        for (int i = 0; i < DIN; ++i) x[i] = ip[i * n0];
#pragma unroll
        for (int i = 0; i < DIN; ++i) F[i] = fx_of(x[i], e);
      } else {
        const int64_t* ip = reinterpret_cast<const int64_t*>(in) + ib;
#pragma unroll
        for (int i = 0; i < DIN; ++i) {
          F[i] = ip[i * n0];
          if (IN == FROM_SUM) F[i] += ip[i * n0 + ks] + ip[i * n0 + 2 * ks];
        }
        if (IN == FROM_SUM) e -= fx_renorm(F);
      }
      fx_core<DIN, DOUT, SYM>(E.f, F, Y);
      if (OUT == TO_DOUBLE) {
        const int X = e + add + 67 - t;
#pragma unroll
        for (int q = 0; q < DOUT; ++q) {
          const double y = fx_store(Y[q], X);
          out[ob + q * n0] = y;
          if (IN == FROM_SUM) m[0] = max(m[0], fx_mag(y));
        }
      } else {
        int64_t* op = reinterpret_cast<int64_t*>(out) + ob;
#pragma unroll
        for (int q = 0; q < DOUT; ++q) op[q * n0] = (int64_t)((uint64_t)Y[q] << sh);
      }
    }
    if (IN == FROM_SUM) block_max<LPB>(omax, 0, min(l, nlines - 1) / LPB, m);
  }
}
template <int N0, int DIN, int DOUT, int SYM, int IN, int OUT, int LPB, int OG = 0, int IBS = 0, int OBS = 0>
__device__ __forceinline__ void chain(const double* in, double* out, EoFp64 E, int nouter, const uint32_t* ex, int add,
                                      int room = 0, int ks = 0, int nex = 1 << 30, uint32_t* omax = nullptr) {
  constexpr uint32_t magic = N0 > 1 ? (uint32_t)((0x100000000ull + N0 - 1) / N0) : 0u;  // l / N0 for l N0 < 2^32
  chain_fp64<DIN, DOUT, SYM, IN, OUT, LPB, LPB / N0, OG, IBS, OBS>(in, ks, out, E, nouter * N0, N0, magic, nex, ex, add, room, omax);
}

// First S^-1 sweep (along x): the sum of three integer arrays V (ks apart; exponent ev + av, two bits free) and of the
// doubles P (largest exponent ep + ap), the one of the smaller exponent shifted down to the other's; then renormalised, to doubles
// with their maxima in omax.
template <int N>
__device__ __noinline__ void chain_sum(const double* V, int ks, const double* P, double* out, EoFp64 E, int nlines,
                                       const uint32_t* ev, int av, const uint32_t* ep, int ap, uint32_t* omax) {
  DGCNS_SHARED(V);
  DGCNS_SHARED(P);
  DGCNS_SHARED(out);
  DGCNS_SHARED(E.f);
  DGCNS_SHARED(ev);
  DGCNS_SHARED(ep);
  const int t = E.f[0].x;
#pragma unroll 1
  for (int l = threadIdx.x; (l & ~31) < nlines; l += blockDim.x) {
    uint32_t m[1] = {0};
    if (l < nlines) {
      const int b = l / (N * N);
      const int xv = fx_exp(ev[b]) + av, xp = fx_exp(ep[b]) + ap + 2, e = max(xv, xp);
      const int sv = min(e - xv, 63);
      const int64_t* v = reinterpret_cast<const int64_t*>(V) + l * N;
      const double* p = P + l * N;
      int64_t F[N], Y[N];
#pragma unroll
      for (int i = 0; i < N; ++i) F[i] = ((v[i] + v[i + ks] + v[i + 2 * ks]) >> sv) + fx_of(p[i], e);
      const int X = e - fx_renorm(F) + 67 - t;
      fx_core<N, N, 1>(E.f, F, Y);
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const double y = fx_store(Y[i], X);
        out[l * N + i] = y;
        m[0] = max(m[0], fx_mag(y));
      }
    }
    block_max<N * N>(omax, 0, min(l, nlines - 1) / (N * N), m);
  }
}

// V_d <- D~_d V_d + the face shares of direction d (lift_body), doubles in, integers out, block exponents ex[cell][5].
template <int N, int D>
__device__ __forceinline__ void chain_lift_dir(double* V, const double* F, EoFp64 E, int nb, bool vol,
                                               const uint32_t* ex) {
  constexpr int N2 = N * N, N3 = N2 * N, st = D == 0 ? 1 : (D == 1 ? N : N2);
  const int sh = E.f[0].y - 2;
#pragma unroll 1
  for (int l = threadIdx.x; l < nb * 5 * N2; l += blockDim.x) {
    const int ec = l / N2, j = l - ec * N2, e = ec / 5, c = ec - 5 * e;
    const double* f0 = F + (size_t)e * (6 * 2 * 5 * N2) + (2 * D * 2 * 5 + c) * N2 + j;
    const double* f1 = f0 + 2 * 5 * N2;
    double x[N + 4];
    x[0] = f0[5 * N2];
    x[1] = f0[0];
    x[N + 2] = -f1[0];
    x[N + 3] = f1[5 * N2];
    double* v = V + ec * N3 + face_node<N>(D, 0, j % N, j / N);
#pragma unroll
    for (int i = 0; i < N; ++i) x[2 + i] = vol ? v[i * st] : 0.0;
    const int E0 = fx_exp(ex[ec]);
    int64_t G[N + 4], Y[N];
#pragma unroll
    for (int i = 0; i < N + 4; ++i) G[i] = fx_of(x[i], E0);
    fx_core<N + 4, N, -1>(E.f, G, Y);
#pragma unroll
    for (int i = 0; i < N; ++i) reinterpret_cast<int64_t*>(v)[i * st] = (int64_t)((uint64_t)Y[i] << sh);
  }
}
template <int N>
__device__ __noinline__ void chain_lift(double* V, const double* F, EoFp64 E, int nb, bool vol, int n3,
                                        const uint32_t* ex) {
  DGCNS_SHARED(V);
  DGCNS_SHARED(E.f);
  DGCNS_SHARED(ex);
  chain_lift_dir<N, 0>(V, F, E, nb, vol, ex);
  chain_lift_dir<N, 1>(V + n3, F, E, nb, vol, ex);
  chain_lift_dir<N, 2>(V + 2 * n3, F, E, nb, vol, ex);
}

}  // namespace dgcns
