// Element Jacobian blocks A, B, C, D of the hybridized stage (Pereira & Vermeire,
// arXiv 2401.16632, Sec. 3.2, eqs. elemA, elemsystem, elemsystemB), for the stage residual
// h = u - u* - a dt R(u, u^) and the element's trace-residual contribution g^k:
//     A = dh/du = I - a dt dR/du,  B = dh/du^ = -a dt dR/du^,  C = dg^k/du,  D = dg^k/du^.
//
// One CTA per implicit element.  The linearisation is organised around the structure of
// the tensor-product operators instead of differentiating the whole element residual:
//   1. exact pointwise Jacobians of the volume flux (w.r.t. the state and the reference
//      gradient) and of the common face flux (w.r.t. face state, trace, face gradient), by
//      forward-mode dual numbers where the flux is nonlinear in the input;
//   2. a seed (a solution point or a trace point) moves the corrected gradient only on the two grid
//      lines through it, and off its own line in proportion to one reference weight, so the bracket
//      of every output along a line is an entry of a small table: full line sums for seeds on the
//      line, single terms for seeds off it;
//   3. every entry of the blocks is one or two table entries times reference weights, written in
//      row order.
// Work per element is O((nA + nT)^2), not the O((nA + nT) x residual) of a dense sweep.
// T = double (plain path) or float (mixed path; blocks stored in FP32).
#include "hfr_internal.h"

namespace hfr {

constexpr int JAC_THREADS = 256;
// resident CTAs per SM asked of the compiler: what the tables of JacWork leave room for
template <typename T>
constexpr int jac_blocks(int p) {
  return sizeof(T) == 4 ? (p <= 3 ? 4 : (p == 4 ? 3 : 2)) : (p <= 3 ? 2 : 1);
}

template <int P, int PHYS, typename T>
struct JacWork {
  static constexpr int N = P + 1, NS = N * N, NV = Phys<PHYS>::NV, NF = 4 * N;
  T U[NS][NV];
  T Uf[NF][NV];
  T ub[NF][NV];
  T un[NF][NV];
  T q[NS][2][NV];
  T qf[NF][2][NV];
  T iJ[NS];
  T Sm[NS][2][2];
  T fJ[NF], fn[NF][2];
  // pointwise Jacobians, innermost index the input variable (read NV-wide: 16-byte aligned)
  alignas(16) T KU[NS][2][NV][NV];
  alignas(16) T KQ[NS][2][2][NV][NV];
  alignas(16) T GU[NF][NV][NV];
  alignas(16) T GH[NF][NV][NV];
  alignas(16) T GQ[NF][2][NV][NV];
  T ciJ[NS];  // a dt / J at each solution point
  // direction d = 0: the xi line (grid row) m, 1: the eta line (grid column) m; position p along it;
  // seed s along it, N and N + 1 the traces at its two ends; entries [v][seed][v0]
  alignas(16) T XT[2][N][N][NV][N][NV];      // flux divergence of a seed off the line, per unit of its weight
  alignas(16) T XF[2][N][N][NV][N + 2][NV];  // ... of a seed on the line
  alignas(16) T HX[4][N][NV][N][NV];         // common face flux of a seed off the line, per unit of its weight
  alignas(16) T FL[4][N][NV][N + 2][NV];     // ... of a seed on the line
  T QO[4][N][N][2], QL[4][N][N + 2][2];      // the face gradients of the same seeds
  T rM[N][N], rdgL[N], rdgR[N], rlm[N], rlp[N], rw[N];  // reference operators in T
  int kf[4];
};

// VW consecutive values: 16 bytes, or one value
template <typename T, int VW>
__device__ __forceinline__ void ldw(const T* p, T (&x)[VW]) {
  if constexpr (VW == 2) {
    const double2 q = *reinterpret_cast<const double2*>(p);
    x[0] = q.x; x[1] = q.y;
  } else {
    ldv<T, VW>(p, x);
  }
}
template <typename T, int VW>
__device__ __forceinline__ void stw(T* p, const T (&x)[VW]) {
  if constexpr (VW == 2) {
    *reinterpret_cast<double2*>(p) = make_double2(x[0], x[1]);
  } else {
    stv<T, VW>(p, x);
  }
}

// total flux F = F^c - F^v at a solution point
template <int PHYS, typename S, typename R, int NV>
__device__ __forceinline__ void vol_flux(const PhysConst<R>& pp, bool visc, const S* u, const S q[2][NV], S F[2][NV]) {
  Phys<PHYS>::template conv<S, R>(pp, u, F);
  if (visc) {
    S Fv[2][NV];
    Phys<PHYS>::template visc<S, R>(pp, u, q, Fv);
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int v = 0; v < NV; ++v) F[c][v] = F[c][v] - Fv[c][v];
  }
}

// common normal flux J_f F^.n of an implicit element's face (trace or IMEX-interface face)
template <int PHYS, typename S, typename R, int NV>
__device__ __forceinline__ void imp_face_flux(const PhysConst<R>& pp, bool visc, int kf, const S* Uf, const S* ub,
                                              const S qf[2][NV], const S* un, R Jf, R n0, R n1, S* Fn) {
  S F[2][NV];
  if (kf == FK_TRACE) {
    Phys<PHYS>::template conv<S, R>(pp, ub, F);
    S s = Phys<PHYS>::template stab<S, R>(pp, ub, n0, n1);
#pragma unroll
    for (int v = 0; v < NV; ++v) Fn[v] = n0 * F[0][v] + n1 * F[1][v] + s * (Uf[v] - ub[v]);
    if (visc) {
      Phys<PHYS>::template visc<S, R>(pp, ub, qf, F);
#pragma unroll
      for (int v = 0; v < NV; ++v) Fn[v] = Fn[v] - (n0 * F[0][v] + n1 * F[1][v]);
    }
  } else {
    S G[2][NV];
    Phys<PHYS>::template conv<S, R>(pp, Uf, F);
    Phys<PHYS>::template conv<S, R>(pp, un, G);
    S lam = dmax(Phys<PHYS>::template wave<S, R>(pp, Uf, n0, n1), Phys<PHYS>::template wave<S, R>(pp, un, n0, n1));
#pragma unroll
    for (int v = 0; v < NV; ++v)
      Fn[v] = R(0.5) * (n0 * (F[0][v] + G[0][v]) + n1 * (F[1][v] + G[1][v])) + R(0.5) * lam * (Uf[v] - un[v]);
    if (visc) {
      Phys<PHYS>::template visc<S, R>(pp, Uf, qf, F);
#pragma unroll
      for (int v = 0; v < NV; ++v) Fn[v] = Fn[v] - (n0 * F[0][v] + n1 * F[1][v]);
    }
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) Fn[v] = Jf * Fn[v];
}

template <int P, int PHYS, typename T>
__global__ void __launch_bounds__(JAC_THREADS, jac_blocks<T>(P)) k_jacobian(const __grid_constant__ RefOps ref,
                                                          const __grid_constant__ PhysParams pp,
                                                          const __grid_constant__ JacArgs a) {
  using W = JacWork<P, PHYS, T>;
  using DT = Dual<T>;
  constexpr int N = W::N, NS = W::NS, NV = W::NV, NF = W::NF;
  constexpr int nA = NS * NV, nT = NF * NV;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  W& w = *reinterpret_cast<W*>(smem_raw);
  const int k = blockIdx.x;
  if (k >= a.Eim) return;
  const int e = a.imp_idx[k];
  const int tid = threadIdx.x;
  const bool visc = phys_viscous(pp);
  const PhysConst<T> pc = phys_const<T>(pp);
  const double* gs = a.geo_sol + (size_t)e * NS * 5;
  const double* gf = a.geo_face + (size_t)e * NF * 3;

  // ---------------------------------------------------------------- primal state (in T)
  for (int i = tid; i < nA; i += JAC_THREADS) w.U[i / NV][i % NV] = T(a.U[(size_t)e * nA + i]);
  for (int i = tid; i < NS; i += JAC_THREADS) {
    w.iJ[i] = T(gs[i * 5]);
    w.ciJ[i] = T(a.a_dt * gs[i * 5]);
    w.Sm[i][0][0] = T(gs[i * 5 + 1]);
    w.Sm[i][0][1] = T(gs[i * 5 + 2]);
    w.Sm[i][1][0] = T(gs[i * 5 + 3]);
    w.Sm[i][1][1] = T(gs[i * 5 + 4]);
  }
  for (int j = tid; j < NF; j += JAC_THREADS) {
    w.fJ[j] = T(gf[j * 3]);
    w.fn[j][0] = T(gf[j * 3 + 1]);
    w.fn[j][1] = T(gf[j * 3 + 2]);
  }
  if (tid < 4) w.kf[tid] = a.kind[e * 4 + tid];
  for (int i = tid; i < N * N; i += JAC_THREADS) w.rM[i / N][i % N] = T(ref.M[i / N][i % N]);
  if (tid < N) {
    w.rdgL[tid] = T(ref.dgL[tid]);
    w.rdgR[tid] = T(ref.dgR[tid]);
    w.rlm[tid] = T(ref.lm[tid]);
    w.rlp[tid] = T(ref.lp[tid]);
    w.rw[tid] = T(ref.w[tid]);
  }
  __syncthreads();
  // one thread per (flux point, variable): face values, then the trace or the neighbour's state
  for (int it = tid; it < NF * NV; it += JAC_THREADS) {
    const int j = it / NV, v = it % NV;
    const int f = j / N, m = j % N, r = f >> 1;
    const T* l = (f & 1) ? w.rlp : w.rlm;
    T s = T(0);
#pragma unroll
    for (int c = 0; c < N; ++c) s += l[c] * w.U[line_pt<N>(r, m, c)][v];
    w.Uf[j][v] = s;
    if (w.kf[f] == FK_TRACE) {
      const int t = (int)FR_IDX(a.tr_of[e * 4 + f], a.ntrace, 23);
      w.ub[j][v] = T(a.uhat[((size_t)t * N + m) * NV + v]);
      w.un[j][v] = s;
    } else {  // interface face: explicit neighbour's state is the common solution
      const int en = (int)FR_IDX(a.nbr[e * 4 + f], a.E, 24), fnb = (int)FR_IDX(a.nbr_face[e * 4 + f], 4, 25);
      const T un = T(a.Uf_all[((size_t)en * NF + fnb * N + m) * NV + v]);
      w.un[j][v] = un;
      w.ub[j][v] = un;
    }
  }
  __syncthreads();
  if (visc) {
    for (int it = tid; it < NS * NV; it += JAC_THREADS) {  // one thread per (point, variable)
      const int i = it / NV, v = it % NV;
      const int ai = i % N, bi = i / N;
      T q0 = w.rdgL[ai] * w.ub[bi][v] + w.rdgR[ai] * w.ub[N + bi][v];
      T q1 = w.rdgL[bi] * w.ub[2 * N + ai][v] + w.rdgR[bi] * w.ub[3 * N + ai][v];
#pragma unroll
      for (int c = 0; c < N; ++c) {
        q0 += w.rM[ai][c] * w.U[c + N * bi][v];
        q1 += w.rM[bi][c] * w.U[ai + N * c][v];
      }
      w.q[i][0][v] = w.iJ[i] * (w.Sm[i][0][0] * q0 + w.Sm[i][1][0] * q1);
      w.q[i][1][v] = w.iJ[i] * (w.Sm[i][0][1] * q0 + w.Sm[i][1][1] * q1);
    }
    __syncthreads();
    for (int it = tid; it < NF * 2 * NV; it += JAC_THREADS) {  // (flux point, direction, variable)
      const int j = it / (2 * NV), c2 = (it / NV) % 2, v = it % NV;
      const int f = j / N, m = j % N, r = f >> 1;
      const T* l = (f & 1) ? w.rlp : w.rlm;
      T s = T(0);
#pragma unroll
      for (int c = 0; c < N; ++c) s += l[c] * w.q[line_pt<N>(r, m, c)][c2][v];
      w.qf[j][c2][v] = s;
    }
  } else {
    for (int i = tid; i < NS * 2 * NV; i += JAC_THREADS) (&w.q[0][0][0])[i] = T(0);
    for (int i = tid; i < NF * 2 * NV; i += JAC_THREADS) (&w.qf[0][0][0])[i] = T(0);
  }
  __syncthreads();

  // the point of position c on line m of direction d
  auto lpt = [](int d, int m, int c) -> int { return d == 0 ? c + N * m : m + N * c; };
  // face gradients: of a unit move of the reference gradient across the line at its point s (QO), of
  // a unit seed s on the line (QL)
  for (int it = tid; it < 4 * N * (2 * N + 2); it += JAC_THREADS) {
    const int s2 = it % (2 * N + 2), m = it / (2 * N + 2) % N, f = it / ((2 * N + 2) * N), d = f >> 1;
    const T* l = (f & 1) ? w.rlp : w.rlm;
    if (s2 < N) {
      const int pt = lpt(d, m, s2);
      const T c = l[s2] * w.iJ[pt];
      w.QO[f][m][s2][0] = c * w.Sm[pt][1 - d][0];
      w.QO[f][m][s2][1] = c * w.Sm[pt][1 - d][1];
    } else {
      const int sd = s2 - N;
      T q0 = T(0), q1 = T(0);
#pragma unroll
      for (int c = 0; c < N; ++c) {
        const int pt = lpt(d, m, c);
        const T wl = l[c] * w.iJ[pt];
        const T wd = wl * (sd < N ? w.rM[c][sd] : (sd == N ? w.rdgL[c] : w.rdgR[c]));
        q0 += wd * w.Sm[pt][d][0];
        q1 += wd * w.Sm[pt][d][1];
        if (c == sd) {
          q0 += wl * w.rM[m][m] * w.Sm[pt][1 - d][0];
          q1 += wl * w.rM[m][m] * w.Sm[pt][1 - d][1];
        }
      }
      w.QL[f][m][sd][0] = q0;
      w.QL[f][m][sd][1] = q1;
    }
  }

  // -------------------------------------------------- 1. pointwise Jacobians
  // volume: items (point, input variable) for the state, then the same for the gradient, each
  // range padded to whole warps so that a warp takes one branch.  Dual numbers only where the flux is
  // nonlinear in the input: the viscous flux is linear in the gradient and the stabilisation in the
  // face state, so those Jacobians are plain evaluations.  In FP64 the pointwise part is the kernel's
  // bound (each warp instruction holds the pipe): with dual numbers for every input, and face items
  // that mixed the kinds within a warp, a stage of 64 x 64 FP64 elements, p = 3, took 29.1 ms; 28.2 now.
  constexpr int NI = (NS * NV + 31) / 32 * 32;
  for (int it = tid; it < 2 * NI; it += JAC_THREADS) {
    const bool isq = it >= NI;
    const int idx = isq ? it - NI : it;
    if (idx >= NS * NV) continue;
    const int i = idx / NV, vp = idx % NV;
    if (!isq) {
      DT u[NV], qd[2][NV], F[2][NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        u[v] = DT(w.U[i][v], v == vp ? T(1) : T(0));
        qd[0][v] = DT(w.q[i][0][v]);
        qd[1][v] = DT(w.q[i][1][v]);
      }
      vol_flux<PHYS, DT, T, NV>(pc, visc, u, qd, F);
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int v = 0; v < NV; ++v) w.KU[i][r][v][vp] = w.Sm[i][r][0] * F[0][v].d + w.Sm[i][r][1] * F[1][v].d;
    } else {
      // only the viscous flux depends on the gradient, and linearly: its value at a unit gradient
      T acc[2][2][NV];
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int r2 = 0; r2 < 2; ++r2)
#pragma unroll
          for (int v = 0; v < NV; ++v) acc[r][r2][v] = T(0);
      if (visc) {
        T u[NV], qe[2][NV], F[2][NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          u[v] = w.U[i][v];
          qe[0][v] = qe[1][v] = T(0);
        }
#pragma unroll
        for (int c2 = 0; c2 < 2; ++c2) {
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            qe[c2][v] = v == vp ? T(1) : T(0);
            qe[1 - c2][v] = T(0);
          }
          Phys<PHYS>::template visc<T, T>(pc, u, qe, F);
#pragma unroll
          for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int v = 0; v < NV; ++v) {
              const T dFr = -(w.Sm[i][r][0] * F[0][v] + w.Sm[i][r][1] * F[1][v]);  // d F~_r / d q_{c2}
#pragma unroll
              for (int r2 = 0; r2 < 2; ++r2) acc[r][r2][v] += dFr * w.iJ[i] * w.Sm[i][r2][c2];
            }
        }
      }
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int r2 = 0; r2 < 2; ++r2)
#pragma unroll
          for (int v = 0; v < NV; ++v) w.KQ[i][r][r2][v][vp] = acc[r][r2][v];
    }
  }
  // face: items (flux point, input variable), each kind of input in whole warps: 0 the trace (dual
  // numbers), 1 the face state (on a trace face the flux moves with it as J_f s 1; interface faces by
  // dual numbers), 2 and 3 the gradient (linear: the viscous flux at a unit gradient)
  constexpr int FI = (NF * NV + 31) / 32 * 32;
  for (int it = tid; it < 4 * FI; it += JAC_THREADS) {
    const int grp = it / FI, idx = it % FI;
    if (idx >= NF * NV) continue;
    const int j = idx / NV, vp = idx % NV;
    const int kf = w.kf[j / N];
    const T n0 = w.fn[j][0], n1 = w.fn[j][1], Jf = w.fJ[j];
    T d[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) d[v] = T(0);
    if (grp >= 2) {
      if (visc) {
        T u[NV], qe[2][NV], F[2][NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          u[v] = kf == FK_TRACE ? w.ub[j][v] : w.Uf[j][v];
          qe[0][v] = (grp == 2 && v == vp) ? T(1) : T(0);
          qe[1][v] = (grp == 3 && v == vp) ? T(1) : T(0);
        }
        Phys<PHYS>::template visc<T, T>(pc, u, qe, F);
#pragma unroll
        for (int v = 0; v < NV; ++v) d[v] = -Jf * (n0 * F[0][v] + n1 * F[1][v]);
      }
    } else if (grp == 1 && kf == FK_TRACE) {
      const T s = Jf * Phys<PHYS>::template stab<T, T>(pc, w.ub[j], n0, n1);
#pragma unroll
      for (int v = 0; v < NV; ++v) d[v] = v == vp ? s : T(0);
    } else if (grp == 1 || kf == FK_TRACE) {
      DT Uf[NV], ub[NV], un[NV], qf[2][NV], Fn[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        Uf[v] = DT(w.Uf[j][v], (grp == 1 && v == vp) ? T(1) : T(0));
        ub[v] = DT(w.ub[j][v], (grp == 0 && v == vp) ? T(1) : T(0));
        un[v] = DT(w.un[j][v]);
        qf[0][v] = DT(w.qf[j][0][v]);
        qf[1][v] = DT(w.qf[j][1][v]);
      }
      imp_face_flux<PHYS, DT, T, NV>(pc, visc, kf, Uf, ub, qf, un, Jf, n0, n1, Fn);
#pragma unroll
      for (int v = 0; v < NV; ++v) d[v] = Fn[v].d;
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      if (grp == 0) w.GH[j][v][vp] = d[v];
      else if (grp == 1) w.GU[j][v][vp] = d[v];
      else w.GQ[j][grp - 2][v][vp] = d[v];
    }
  }
  __syncthreads();

  // ------------------------------------------------ 2. tables of the lines
  // A unit seed at the solution point (a0, b0) or on a trace moves the reference gradient only on its
  // grid row and column:
  //   dR(ai, bi) = -1/J [ sum_c M[ai][c] dFx(c, bi) - dgL[ai] dFn(xi-, bi) + dgR[ai] dFn(xi+, bi)
  //                     + the same along eta ]
  // On the row bi = b0 the xi bracket is a full line sum (XF[0][b0][ai][a0]).  On any other row only
  // the point (a0, bi) moves, by its eta reference gradient M[bi][b0], and the two face points of
  // that row with it: the bracket is M[bi][b0] times a table without b0 (XT[0][bi][ai][a0]).  The eta
  // bracket likewise, with the columns; a trace seed replaces M[.][a0] by dgL or dgR.  So every
  // output of A, B, C and D is a table entry times a reference weight, or the sum of two.
  // Bound by the stores of the blocks, 130 KB per element at p = 4.  One seed point per warp with
  // the tangents of its two lines, six vector reads of shared memory per output vector, kept the
  // shared-memory pipe at 89 %: 368 us for 4096 elements, p = 4, FP32 (the blocks alone take 79 us
  // at the copy rate); 195 us by the tables.  FP64, p = 3: 1.65 ms, 1.0 ms now.
  constexpr int CI = N * NV * (2 * N + 2);
  for (int it = tid; it < 4 * CI; it += JAC_THREADS) {
    const int f = it / CI, s2 = it % (2 * N + 2), v = it / (2 * N + 2) % NV, m = it / ((2 * N + 2) * NV) % N;
    const int j = f * N + m;
    T g0[NV], g1[NV], o[NV];
    ldv<T, NV>(&w.GQ[j][0][v][0], g0);
    ldv<T, NV>(&w.GQ[j][1][v][0], g1);
    const T q0 = s2 < N ? w.QO[f][m][s2][0] : w.QL[f][m][s2 - N][0];
    const T q1 = s2 < N ? w.QO[f][m][s2][1] : w.QL[f][m][s2 - N][1];
#pragma unroll
    for (int x = 0; x < NV; ++x) o[x] = g0[x] * q0 + g1[x] * q1;
    if (s2 < N) {
      stv<T, NV>(&w.HX[f][m][v][s2][0], o);
    } else {
      const int sd = s2 - N;
      if (sd < N) {
        const T l = (f & 1) ? w.rlp[sd] : w.rlm[sd];
        ldv<T, NV>(&w.GU[j][v][0], g0);
#pragma unroll
        for (int x = 0; x < NV; ++x) o[x] += g0[x] * l;
      } else if (w.kf[(f & 2) + sd - N] != FK_TRACE) {
#pragma unroll
        for (int x = 0; x < NV; ++x) o[x] = T(0);
      } else if (sd - N == (f & 1)) {
        ldv<T, NV>(&w.GH[j][v][0], g0);
#pragma unroll
        for (int x = 0; x < NV; ++x) o[x] += g0[x];
      }
      stv<T, NV>(&w.FL[f][m][v][sd][0], o);
    }
  }
  __syncthreads();
  // XF items (line, v, seed), then XT items, each kind in whole warps; all positions p of the line
  constexpr int FI2 = (2 * N * NV * (N + 2) + 31) / 32 * 32;
  for (int it = tid; it < FI2 + 2 * N * NV * N; it += JAC_THREADS) {
    const bool full = it < FI2;
    const int idx = full ? it : it - FI2;
    if (full && idx >= 2 * N * NV * (N + 2)) continue;
    const int S1 = full ? N + 2 : N;
    const int sd = idx % S1, v = idx / S1 % NV, m = idx / (S1 * NV) % N, d = idx / (S1 * NV * N);
    T h0[NV], h1[NV], e[NV], t[N][NV];
    if (full) {
      ldv<T, NV>(&w.FL[2 * d][m][v][sd][0], h0);
      ldv<T, NV>(&w.FL[2 * d + 1][m][v][sd][0], h1);
    } else {
      ldv<T, NV>(&w.HX[2 * d][m][v][sd][0], h0);
      ldv<T, NV>(&w.HX[2 * d + 1][m][v][sd][0], h1);
    }
    if (sd < N) {
      const int pt = lpt(d, m, sd);
      ldv<T, NV>(&w.KQ[pt][d][1 - d][v][0], e);
      if (full) {
        T ku[NV];
        ldv<T, NV>(&w.KU[pt][d][v][0], ku);
        const T mm = w.rM[m][m];
#pragma unroll
        for (int x = 0; x < NV; ++x) e[x] = mm * e[x] + ku[x];
      }
    } else {
#pragma unroll
      for (int x = 0; x < NV; ++x) e[x] = T(0);
    }
    if (full) {
      const bool on = sd < N || w.kf[2 * d + sd - N] == FK_TRACE;
#pragma unroll
      for (int c = 0; c < N; ++c) {
        ldv<T, NV>(&w.KQ[lpt(d, m, c)][d][d][v][0], t[c]);
        const T wc = sd < N ? w.rM[c][sd] : (on ? (sd == N ? w.rdgL[c] : w.rdgR[c]) : T(0));
#pragma unroll
        for (int x = 0; x < NV; ++x) t[c][x] *= wc;
      }
    }
#pragma unroll 1
    for (int p = 0; p < N; ++p) {
      T o[NV];
      const T me = sd < N ? w.rM[p][sd] : T(0), gl = w.rdgL[p], gr = w.rdgR[p], cj = w.ciJ[lpt(d, m, p)];
#pragma unroll
      for (int x = 0; x < NV; ++x) o[x] = me * e[x] - gl * h0[x] + gr * h1[x];
      if (full) {
#pragma unroll
        for (int c = 0; c < N; ++c) {
          const T mc = w.rM[p][c];
#pragma unroll
          for (int x = 0; x < NV; ++x) o[x] += mc * t[c][x];
        }
      }
#pragma unroll
      for (int x = 0; x < NV; ++x) o[x] *= cj;  // A = I - a dt dR, B = -a dt dR
      stv<T, NV>(full ? &w.XF[d][m][p][v][sd][0] : &w.XT[d][m][p][v][sd][0], o);
    }
  }
  __syncthreads();

  // ------------------------------------------------ 3. outputs
  // A thread keeps its column group (VW seed variables of one seed) and steps through the rows:
  // consecutive threads write consecutive 16-byte groups.
  constexpr int VW = NV % (16 / (int)sizeof(T)) == 0 ? 16 / (int)sizeof(T) : 1;
  constexpr int CA = nA / VW, CB = nT / VW, RA = JAC_THREADS / CA, RB = JAC_THREADS / CB;
  T* A = reinterpret_cast<T*>(a.A) + (size_t)k * nA * nA;
  T* B = reinterpret_cast<T*>(a.B) + (size_t)k * nA * nT;
  T* C = reinterpret_cast<T*>(a.C) + (size_t)k * nT * nA;
  T* Dm = reinterpret_cast<T*>(a.D) + (size_t)k * nT * nT;
  if (tid < RA * CA) {  // seeds: solution points
    const int cg = tid % CA, sp = cg * VW / NV, v0 = cg * VW % NV, a0 = sp % N, b0 = sp / N;
    for (int i = tid / CA; i < nA; i += RA) {
      const int pt = i / NV, v = i % NV, ai = pt % N, bi = pt / N;
      const bool xrow = bi == b0, ycol = ai == a0;
      const T fx = xrow ? T(1) : w.rM[bi][b0], fy = ycol ? T(1) : w.rM[ai][a0];
      T x[VW], y[VW];
      ldw<T, VW>(xrow ? &w.XF[0][bi][ai][v][a0][v0] : &w.XT[0][bi][ai][v][a0][v0], x);
      ldw<T, VW>(ycol ? &w.XF[1][ai][bi][v][b0][v0] : &w.XT[1][ai][bi][v][b0][v0], y);
#pragma unroll
      for (int u = 0; u < VW; ++u) {
        x[u] = fx * x[u] + fy * y[u];
        if (pt == sp && v == v0 + u) x[u] += T(1);
      }
      stw<T, VW>(A + (size_t)i * nA + cg * VW, x);
    }
    for (int i = tid / CA; i < nT; i += RA) {
      const int j = i / NV, v = i % NV, m = j % N, f = j / N;
      const bool tr = w.kf[f] == FK_TRACE, eta = f >= 2;
      const int sl = eta ? b0 : a0, so = eta ? a0 : b0;  // the seed's place along the line, its line
      const bool on = m == so;
      T x[VW];
      ldw<T, VW>(on ? &w.FL[f][m][v][sl][v0] : &w.HX[f][m][v][sl][v0], x);
      const T c = on ? w.rw[m] : w.rw[m] * w.rM[m][so];
#pragma unroll
      for (int u = 0; u < VW; ++u) x[u] = tr ? c * x[u] : T(0);
      stw<T, VW>(C + (size_t)i * nA + cg * VW, x);
    }
  }
  if (tid < RB * CB) {  // seeds: trace points
    const int cg = tid % CB, j0 = cg * VW / NV, v0 = cg * VW % NV, f0 = j0 / N, m0 = j0 % N;
    const int d0 = f0 >> 1, sd = N + (f0 & 1);
    const bool act = w.kf[f0] == FK_TRACE;
    const T* dgs = (f0 & 1) ? w.rdgR : w.rdgL;
    for (int i = tid / CB; i < nA; i += RB) {
      const int pt = i / NV, v = i % NV, ai = pt % N, bi = pt / N;
      const int p = d0 ? bi : ai, m = d0 ? ai : bi;  // the point on the lines along the seed's direction
      T x[VW], y[VW];
      ldw<T, VW>(&w.XT[1 - d0][p][m][v][m0][v0], y);
      const T fy = act ? dgs[p] : T(0);
#pragma unroll
      for (int u = 0; u < VW; ++u) x[u] = act ? fy * y[u] : T(0);
      if (act && m == m0) {
        ldw<T, VW>(&w.XF[d0][m][p][v][sd][v0], y);
#pragma unroll
        for (int u = 0; u < VW; ++u) x[u] += y[u];
      }
      stw<T, VW>(B + (size_t)i * nT + cg * VW, x);
    }
    for (int i = tid / CB; i < nT; i += RB) {
      const int j = i / NV, v = i % NV, m = j % N, f = j / N;
      const bool same = (f >> 1) == d0;
      const bool nz = act && w.kf[f] == FK_TRACE && (!same || m == m0);
      T x[VW];
      ldw<T, VW>(same ? &w.FL[f][m][v][sd][v0] : &w.HX[f][m][v][m0][v0], x);
      const T c = same ? w.rw[m] : w.rw[m] * dgs[m];
#pragma unroll
      for (int u = 0; u < VW; ++u) x[u] = nz ? c * x[u] : T(0);
      stw<T, VW>(Dm + (size_t)i * nT + cg * VW, x);
    }
  }
}

template <int P, int PHYS, typename T>
static cudaError_t jac_impl(const RefOps& ref, const PhysParams& pp, const JacArgs& a, cudaStream_t st) {
  size_t smem = sizeof(JacWork<P, PHYS, T>);
  auto kern = k_jacobian<P, PHYS, T>;
  cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  // several CTAs per SM: ask for the largest shared-memory carveout
  err = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  if (err != cudaSuccess) return err;
  if (a.Eim == 0) return cudaSuccess;
  (hfr::count_launch(), kern<<<a.Eim, JAC_THREADS, smem, st>>>(ref, pp, a));
  return cudaGetLastError();
}

template <typename T>
static cudaError_t jac_dispatch(int p, const RefOps& ref, const PhysParams& pp, const JacArgs& a, cudaStream_t st) {
  if (pp.kind == 0) {
    switch (p) {
      case 1: return jac_impl<1, 0, T>(ref, pp, a, st);
      case 2: return jac_impl<2, 0, T>(ref, pp, a, st);
      case 3: return jac_impl<3, 0, T>(ref, pp, a, st);
    }
  } else if (pp.kind == 2) {
    switch (p) {
      case 2: return jac_impl<2, 2, T>(ref, pp, a, st);
      case 3: return jac_impl<3, 2, T>(ref, pp, a, st);
      case 4: return jac_impl<4, 2, T>(ref, pp, a, st);
    }
  } else {
    switch (p) {
      case 2: return jac_impl<2, 1, T>(ref, pp, a, st);
      case 3: return jac_impl<3, 1, T>(ref, pp, a, st);
      case 4: return jac_impl<4, 1, T>(ref, pp, a, st);
      case 5: return jac_impl<5, 1, T>(ref, pp, a, st);
    }
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_jacobian(int p, int prec_bytes, const RefOps& ref, const PhysParams& pp, const JacArgs& a,
                            cudaStream_t st) {
  if (prec_bytes == 8) return jac_dispatch<double>(p, ref, pp, a, st);
  return jac_dispatch<float>(p, ref, pp, a, st);
}

}  // namespace hfr

#include "hfr_checked_unit.inc"
