// Hexahedral elements of the general-mesh path: the FR / hybridized-FR residual and the element
// blocks in three dimensions (Pereira & Vermeire, arXiv 2401.16632: the scheme of Secs. 2-4, run
// on hexahedra in Sec. 5.3; compressible Navier-Stokes with u = (rho, rho v, E)).
//
// The 2D operators in tensor product: solution point pt = a + n b + n^2 c; face f has normal axis
// r = f / 2 and side sigma (f odd: +1); face point m = i + n j along the lower then the higher
// tangential axis; the line of solution points through face point m along r is
//     r = 0: s + n i + n^2 j,   r = 1: i + n s + n^2 j,   r = 2: i + n j + n^2 s   (s = 0..n-1).
// With the 1D lift l_s(+-1)/w_s of the DG-recovering corrections folded into
// M = D - dgL lm^T - dgR lp^T (as in two dimensions):
//     Q_r(pt) = sum_s M[a_r][s] U(line) + dgL[a_r] u_bar(face 2r) + dgR[a_r] u_bar(face 2r+1)
//     q_c     = (1/J) sum_r S[r][c] Q_r,            S[r] = x_{xi_s} x x_{xi_t} (cyclic (r, s, t))
//     R       = -(1/J) sum_r [sum_s M[a_r][s] F~_r(line) - dgL[a_r] Fn(2r) + dgR[a_r] Fn(2r+1)]
// where a_r is the point's index along r and Fn = J_f F^.n the common normal flux at the face
// point met by the point's r-line.  Face kinds, common fluxes, trace rows and the viscous readings
// are those of the quadrilateral path (one degree: face points are the element's face nodes).
//
// Element blocks are formed column by column (one warp per seed point, tangents along the seed's
// grid lines) and stored column-major, so that a warp writes its columns as contiguous runs.
#include <math.h>
#include <string.h>

#include "hfr_general_internal.h"

namespace hfr {
namespace gen {

constexpr int HN = HEX_PMAX + 1;       // points per line (at most)
constexpr int HNS = HN * HN * HN;      // solution points
constexpr int HNF = HN * HN;           // points per face
constexpr int HFP = 6 * HNF;           // face points per element
constexpr int HNV = 5;
constexpr int HT = 128;                // threads of the residual kernel (one CTA per element)

// Navier-Stokes in three dimensions (ideal gas, R = 1, constant mu, Stokes hypothesis,
// kappa = mu gamma / ((gamma - 1) Pr)); F[c][v], q[c][v] = du_v / dx_c
struct NS3 {
  template <typename S, typename R>
  __device__ static void conv(const PhysConst<R>& pc, const S* u, S F[3][HNV]) {
    const S ir = R(1) / u[0];
    const S v0 = u[1] * ir, v1 = u[2] * ir, v2 = u[3] * ir;
    const S p = pc.gm1 * (u[4] - R(0.5) * (u[1] * v0 + u[2] * v1 + u[3] * v2));
    const S v[3] = {v0, v1, v2};
    const S Ep = u[4] + p;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      F[c][0] = u[1 + c];
#pragma unroll
      for (int k = 0; k < 3; ++k) F[c][1 + k] = u[1 + k] * v[c] + (k == c ? p : S(R(0)));
      F[c][4] = Ep * v[c];
    }
  }
  template <typename S, typename R>
  __device__ static void visc(const PhysConst<R>& pc, const S* u, const S q[3][HNV], S F[3][HNV]) {
    const R mu = pc.mu;
    const S ir = R(1) / u[0];
    const S v[3] = {u[1] * ir, u[2] * ir, u[3] * ir};
    const S e = u[4] * ir;
    S dv[3][3], dT[3];  // dv[c][k] = d v_k / d x_c
#pragma unroll
    for (int c = 0; c < 3; ++c) {
#pragma unroll
      for (int k = 0; k < 3; ++k) dv[c][k] = (q[c][1 + k] - v[k] * q[c][0]) * ir;
      dT[c] = pc.gm1 * ((q[c][4] - e * q[c][0]) * ir - (v[0] * dv[c][0] + v[1] * dv[c][1] + v[2] * dv[c][2]));
    }
    const S div = dv[0][0] + dv[1][1] + dv[2][2];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      F[c][0] = S(R(0));
#pragma unroll
      for (int k = 0; k < 3; ++k) F[c][1 + k] = mu * (dv[c][k] + dv[k][c] - (k == c ? R(2.0 / 3.0) * div : S(R(0))));
      F[c][4] = v[0] * F[c][1] + v[1] * F[c][2] + v[2] * F[c][3] + pc.kappa * dT[c];
    }
  }
  template <typename S, typename R>
  __device__ static S wave(const PhysConst<R>& pc, const S* u, const R* n) {
    const S ir = R(1) / u[0];
    const S v0 = u[1] * ir, v1 = u[2] * ir, v2 = u[3] * ir;
    const S p = pc.gm1 * (u[4] - R(0.5) * (u[1] * v0 + u[2] * v1 + u[3] * v2));
    return dabs(v0 * n[0] + v1 * n[1] + v2 * n[2]) + dsqrt(pc.gamma * p * ir);
  }
  template <typename S, typename R>
  __device__ static S stab(const PhysConst<R>& pc, const S* u, const R* n) {
    return wave<S, R>(pc, u, n) + pc.mu_lref / u[0];
  }
};

// common normal flux J_f F^.n and the trace row of one face point (as gface_flux in 2D)
template <typename S, typename R>
__device__ __forceinline__ void hface_flux(const PhysConst<R>& pc, bool visc, int kf, bool traced, bool imp,
                                           const S* uf, const S* ub, const S (&qf)[3][HNV], const S* un,
                                           const S (&qn)[3][HNV], R Jf, const R* nr, const R* uinf, S* Fn, S* row) {
  S F[3][HNV];
  if (traced) {
    S Fh[HNV];
    NS3::conv<S, R>(pc, ub, F);
    const S s = NS3::stab<S, R>(pc, ub, nr);
#pragma unroll
    for (int v = 0; v < HNV; ++v) Fh[v] = nr[0] * F[0][v] + nr[1] * F[1][v] + nr[2] * F[2][v] + s * (uf[v] - ub[v]);
    if (visc) {
      NS3::visc<S, R>(pc, ub, qf, F);
#pragma unroll
      for (int v = 0; v < HNV; ++v) Fh[v] = Fh[v] - (nr[0] * F[0][v] + nr[1] * F[1][v] + nr[2] * F[2][v]);
    }
#pragma unroll
    for (int v = 0; v < HNV; ++v) Fn[v] = Jf * Fh[v];
    if (kf == FK_FAR) {
#pragma unroll
      for (int v = 0; v < HNV; ++v) row[v] = Jf * s * ((uf[v] - ub[v]) + (uinf[v] - ub[v]));
    } else if (kf == FK_WALL) {
#pragma unroll
      for (int v = 0; v < HNV; ++v) row[v] = (v == 0 || v == HNV - 1) ? Jf * Fh[v] : Jf * s * ub[v];
    } else {
#pragma unroll
      for (int v = 0; v < HNV; ++v) row[v] = Jf * Fh[v];
    }
    return;
  }
  S G[3][HNV];
  NS3::conv<S, R>(pc, uf, F);
  NS3::conv<S, R>(pc, un, G);
  const S lam = dmax(NS3::wave<S, R>(pc, uf, nr), NS3::wave<S, R>(pc, un, nr));
  S Fh[HNV];
#pragma unroll
  for (int v = 0; v < HNV; ++v)
    Fh[v] = R(0.5) * (nr[0] * (F[0][v] + G[0][v]) + nr[1] * (F[1][v] + G[1][v]) + nr[2] * (F[2][v] + G[2][v])) +
            R(0.5) * lam * (uf[v] - un[v]);
  if (visc) {
    if (kf == FK_FR || kf == FK_FAR) {
      NS3::visc<S, R>(pc, uf, qf, F);
      NS3::visc<S, R>(pc, un, qn, G);
#pragma unroll
      for (int v = 0; v < HNV; ++v)
        Fh[v] = Fh[v] - R(0.5) * (nr[0] * (F[0][v] + G[0][v]) + nr[1] * (F[1][v] + G[1][v]) + nr[2] * (F[2][v] + G[2][v]));
    } else {
      if (imp)
        NS3::visc<S, R>(pc, uf, qf, F);
      else
        NS3::visc<S, R>(pc, un, qn, F);
#pragma unroll
      for (int v = 0; v < HNV; ++v) Fh[v] = Fh[v] - (nr[0] * F[0][v] + nr[1] * F[1][v] + nr[2] * F[2][v]);
    }
  }
#pragma unroll
  for (int v = 0; v < HNV; ++v) {
    Fn[v] = Jf * Fh[v];
    row[v] = S(R(0));
  }
}

// solution point on the r-line through face point m at coordinate s
__device__ __forceinline__ int hline(int r, int m, int s, int n) {
  const int i = m % n, j = m / n;
  return r == 0 ? s + n * i + n * n * j : (r == 1 ? i + n * s + n * n * j : i + n * j + n * n * s);
}
// a point's index along axis r and the face point of its r-line
__device__ __forceinline__ int hcoord(int pt, int r, int n) { return r == 0 ? pt % n : (r == 1 ? (pt / n) % n : pt / (n * n)); }
__device__ __forceinline__ int hfacept(int pt, int r, int n) {
  const int a = pt % n, b = (pt / n) % n, c = pt / (n * n);
  return r == 0 ? b + n * c : (r == 1 ? a + n * c : a + n * b);
}

// ------------------------------------------------------------------------ residual passes
struct HWork {
  double U[HNS][HNV];
  double Uf[HFP][HNV], ub[HFP][HNV];
  double q[HNS][3][HNV];
  double qf[HFP][3][HNV];
  double Ft[HNS][3][HNV];
  double Fn[HFP][HNV];
  double M[HN][HN], lm[HN], lp[HN], dgL[HN], dgR[HN], w[HN];
  int kf[6], tr[6];
};
static_assert(sizeof(HWork) <= 227 * 1024, "hexahedral residual workspace exceeds shared memory");

template <int MODE>
__global__ void __launch_bounds__(HT) k_hex_elem(const __grid_constant__ PhysParams pp, const __grid_constant__ GArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  HWork& w = *reinterpret_cast<HWork*>(smem_raw);
  if ((int)blockIdx.x >= (a.elist ? a.nlist : a.E)) return;
  const int e = a.elist ? a.elist[blockIdx.x] : (int)blockIdx.x;
  const int tid = threadIdx.x;
  const int n = a.deg[e], ns = n * n * n, nf = n * n, FS = a.fs;
  const GenRef& RF = *a.ref;
  const bool visc = phys_viscous(pp);
  const PhysConst<double> pc = phys_const<double>(pp);
  const bool imp = a.implicit[e] != 0;
  for (int i = tid; i < n * n; i += HT) w.M[i / n][i % n] = RF.M[n][i / n][i % n];
  if (tid < n) {
    w.lm[tid] = RF.lm[n][tid];
    w.lp[tid] = RF.lp[n][tid];
    w.dgL[tid] = RF.dgL[n][tid];
    w.dgR[tid] = RF.dgR[n][tid];
    w.w[tid] = RF.w[n][tid];
  }
  if (tid < 6) {
    w.kf[tid] = a.kind[6 * e + tid];
    w.tr[tid] = a.tr_of[6 * e + tid];
  }
  const double* Ue = a.U + a.uoff[e];
  for (int i = tid; i < ns * HNV; i += HT) w.U[i / HNV][i % HNV] = Ue[i];
  __syncthreads();
  // face values
  for (int it = tid; it < 6 * nf * HNV; it += HT) {
    const int f = it / (nf * HNV), m = (it / HNV) % nf, v = it % HNV, r = f >> 1;
    const double* l = (f & 1) ? w.lp : w.lm;
    double s = 0.0;
    for (int c = 0; c < n; ++c) s += l[c] * w.U[hline(r, m, c, n)][v];
    w.Uf[f * nf + m][v] = s;
    if (MODE == GM_UF) a.Uf_out[((size_t)(6 * e + f) * FS + m) * HNV + v] = s;
  }
  if (MODE == GM_UF) return;
  __syncthreads();
  for (int it = tid; it < 6 * nf * HNV; it += HT) {
    const int f = it / (nf * HNV), m = (it / HNV) % nf, v = it % HNV;
    const int kf = w.kf[f], t = w.tr[f];
    const double uf = w.Uf[f * nf + m][v];
    double ub;
    if (t >= 0) {
      ub = a.uhat[(size_t)FR_IDX(a.fnode[(6 * e + f) * FS + m], a.npts, 10) * HNV + v];
    } else if (kf == FK_FAR) {
      ub = 0.5 * (uf + a.uinf[v]);
    } else {
      const int nb = (int)FR_IDX(a.nbr[6 * e + f], a.E, 11), fn = (int)FR_IDX(a.nbr_face[6 * e + f], 6, 12);
      const double un = a.Uf_all[((size_t)(6 * nb + fn) * FS + m) * HNV + v];
      ub = kf == FK_FR ? 0.5 * (uf + un) : (imp ? un : uf);
    }
    w.ub[f * nf + m][v] = ub;
  }
  __syncthreads();
  const double* gs = a.geo_sol + (size_t)a.goff[e] * 10;
  if (visc) {
    for (int it = tid; it < ns * HNV; it += HT) {
      const int i = it / HNV, v = it % HNV;
      double Q[3];
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        const int ar = hcoord(i, r, n), m = hfacept(i, r, n);
        double s = w.dgL[ar] * w.ub[(2 * r) * nf + m][v] + w.dgR[ar] * w.ub[(2 * r + 1) * nf + m][v];
        for (int c = 0; c < n; ++c) s += w.M[ar][c] * w.U[hline(r, m, c, n)][v];
        Q[r] = s;
      }
      const double* G = gs + i * 10;
#pragma unroll
      for (int c = 0; c < 3; ++c) w.q[i][c][v] = G[0] * (G[1 + c] * Q[0] + G[4 + c] * Q[1] + G[7 + c] * Q[2]);
    }
    __syncthreads();
    for (int it = tid; it < 6 * nf * 3 * HNV; it += HT) {
      const int f = it / (nf * 3 * HNV), m = (it / (3 * HNV)) % nf, c2 = (it / HNV) % 3, v = it % HNV, r = f >> 1;
      const double* l = (f & 1) ? w.lp : w.lm;
      double s = 0.0;
      for (int c = 0; c < n; ++c) s += l[c] * w.q[hline(r, m, c, n)][c2][v];
      w.qf[f * nf + m][c2][v] = s;
      if (MODE == GM_QF) a.qf_out[(((size_t)(6 * e + f) * FS + m) * 3 + c2) * HNV + v] = s;
    }
  } else if (MODE == GM_QF) {
    for (int it = tid; it < 6 * FS * 3 * HNV; it += HT) a.qf_out[(size_t)(6 * e) * FS * 3 * HNV + it] = 0.0;
  }
  if (MODE == GM_QF) return;
  __syncthreads();
  for (int i = tid; i < ns; i += HT) {
    const double* G = gs + i * 10;
    double F[3][HNV];
    NS3::conv<double, double>(pc, w.U[i], F);
    if (visc) {
      double Fv[3][HNV];
      NS3::visc<double, double>(pc, w.U[i], w.q[i], Fv);
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int v = 0; v < HNV; ++v) F[c][v] -= Fv[c][v];
    }
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int v = 0; v < HNV; ++v) w.Ft[i][r][v] = G[1 + 3 * r] * F[0][v] + G[2 + 3 * r] * F[1][v] + G[3 + 3 * r] * F[2][v];
  }
  for (int jj = tid; jj < 6 * nf; jj += HT) {
    const int f = jj / nf, m = jj % nf;
    const int kf = w.kf[f];
    const bool traced = w.tr[f] >= 0;
    const double* G = a.geo_face + ((size_t)(6 * e + f) * FS + m) * 4;
    double un[HNV], qn[3][HNV], qf[3][HNV], Fn[HNV], row[HNV];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int v = 0; v < HNV; ++v) qf[c][v] = visc ? w.qf[jj][c][v] : 0.0;
    if (!traced && kf != FK_FAR) {
      const int nb = (int)FR_IDX(a.nbr[6 * e + f], a.E, 11), fn = (int)FR_IDX(a.nbr_face[6 * e + f], 6, 12);
      const size_t nix = (size_t)(6 * nb + fn) * FS + m;
#pragma unroll
      for (int v = 0; v < HNV; ++v) {
        un[v] = a.Uf_all[nix * HNV + v];
#pragma unroll
        for (int c = 0; c < 3; ++c) qn[c][v] = visc ? a.qf_all[(nix * 3 + c) * HNV + v] : 0.0;
      }
    } else {
#pragma unroll
      for (int v = 0; v < HNV; ++v) {
        un[v] = a.uinf[v];
#pragma unroll
        for (int c = 0; c < 3; ++c) qn[c][v] = qf[c][v];
      }
    }
    const double nr[3] = {G[1], G[2], G[3]};
    hface_flux<double, double>(pc, visc, kf, traced, imp, w.Uf[jj], w.ub[jj], qf, un, qn, G[0], nr, a.uinf, Fn, row);
#pragma unroll
    for (int v = 0; v < HNV; ++v) w.Fn[jj][v] = Fn[v];
    if (a.gview) {
      const double wq = traced ? w.w[m % n] * w.w[m / n] : 0.0;
#pragma unroll
      for (int v = 0; v < HNV; ++v) a.gview[((size_t)(6 * e + f) * FS + m) * HNV + v] = wq * row[v];
    }
  }
  __syncthreads();
  for (int it = tid; it < ns * HNV; it += HT) {
    const int i = it / HNV, v = it % HNV;
    double d = 0.0;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const int ar = hcoord(i, r, n), m = hfacept(i, r, n);
      d += -w.dgL[ar] * w.Fn[(2 * r) * nf + m][v] + w.dgR[ar] * w.Fn[(2 * r + 1) * nf + m][v];
      for (int c = 0; c < n; ++c) d += w.M[ar][c] * w.Ft[hline(r, m, c, n)][r][v];
    }
    if (a.R) a.R[a.uoff[e] + it] = -gs[i * 10] * d;
  }
}

cudaError_t hex_elem_pass(GenCtx* g, const GArgs& a, int mode) {
  const size_t smem = sizeof(HWork);
  cudaError_t e;
  auto kern = mode == GM_UF ? k_hex_elem<GM_UF> : (mode == GM_QF ? k_hex_elem<GM_QF> : k_hex_elem<GM_RES>);
  if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
  const int cnt = a.elist ? a.nlist : a.E;
  if (cnt == 0) return cudaSuccess;
  (count_launch(), kern<<<cnt, HT, smem, g->st>>>(g->pp, a));
  return cudaGetLastError();
}

// ------------------------------------------------------------------------ element blocks
// One CTA per implicit element at a time.  Primal state, pointwise Jacobians by dual numbers, then
// one warp per seed point (a solution point or a trace face point: HNV columns).  A seed moves the
// reference gradient on the three grid lines through its point (a trace seed on the one line normal
// to its face), so
//   * the line through an output point along axis r meets them in one point at most, unless it is
//     itself one of them: one product M dQ KQ per axis, or a line sum RC formed once per seed;
//   * the face fluxes move at the 2N - 1 points of a face whose normal lines meet the seed's lines;
//   * every other entry of the columns is zero (27 of 64 points and 54 of 96 face points at N = 4).
// Lane = output row (coalesced column-major stores), HNV seed variables per lane.
//
// The pointwise Jacobians of an FP32 element (33 600 values at N = 4) stay in shared memory; in a
// global slab per CTA, with every tangent of every point formed for each of the 800 columns, the
// kernel took 21.8 ms on 4608 elements of N = 4; it takes 6.6 ms, bound by instruction issue (11.8 GB
// of blocks are 1.7 ms of HBM).  FP64 keeps the slab (268 KB).
template <typename T, int N>
struct HJac {  // innermost index the input variable
  static constexpr int NS = N * N * N, FP = 6 * N * N;
  T KU[NS][3][HNV][HNV];
  T KQ[NS][3][3][HNV][HNV];
  T GU[FP][HNV][HNV], GH[FP][HNV][HNV], GQ[FP][3][HNV][HNV];
  T RH[FP][HNV][HNV];  // boundary faces: the trace row by the trace
};
template <typename T, int N>
struct HJWork {
  static constexpr int NS = N * N * N, NF = N * N, FP = 6 * NF;
  static constexpr int NW = sizeof(T) == 4 ? 12 : 8;  // warps of the CTA
  T iJ[NS], ciJ[NS], Sm[NS][3][3], RU[FP];  // RU: far field, the row by the state (RU 1)
  T M[N][N], lm[N], lp[N], dgL[N], dgR[N], wq[NF], uinf[5];
  int kf[6], tr[6];
  struct Primal {
    T U[NS][HNV];
    T Uf[FP][HNV], ub[FP][HNV], un[FP][HNV];
    T q[NS][3][HNV];
    T qf[FP][3][HNV];
    T fJ[FP], fnr[FP][3];
  };
  struct Col {  // tangents of one seed point, entries [v][v0]
    T RC[3][N][HNV][HNV];       // line sums sum_s M[i][s] dF_r
    T FN[6][2 * N][HNV][HNV];   // face fluxes at the active points (slots of hslot)
    T SD[3][HNV][HNV];          // dF_r at the seed point itself
    T DQ[3][N][3];              // physical gradient tangents on the lines
    T qf[6][2 * N][3];          // gradient tangents at the active face points
  };
  union {
    Primal pr;
    Col col[NW];
  };
};
template <typename T, int N>
constexpr size_t hex_jac_smem() {
  return sizeof(HJWork<T, N>) + (sizeof(T) == 4 ? sizeof(HJac<T, N>) : 0);
}
static_assert(hex_jac_smem<float, HN>() <= 227 * 1024 && hex_jac_smem<double, HN>() <= 227 * 1024,
              "hexahedral block workspace exceeds shared memory");

template <typename T, int N>
__global__ void __launch_bounds__(32 * HJWork<T, N>::NW, 1) k_hex_jacobian(const __grid_constant__ PhysParams pp,
                                                                         const __grid_constant__ GArgs a,
                                                                         const __grid_constant__ JArgs j) {
  using DT = Dual<T>;
  using W = HJWork<T, N>;
  constexpr int ns = W::NS, nf = W::NF, NW = W::NW, NT = 32 * NW;
  constexpr int nA = ns * HNV, nT = 6 * nf * HNV;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  W& w = *reinterpret_cast<W*>(smem_raw);
  HJac<T, N>& J = sizeof(T) == 4 ? *reinterpret_cast<HJac<T, N>*>(smem_raw + sizeof(W))
                                 : reinterpret_cast<HJac<T, N>*>(j.scratch)[blockIdx.x];
  typename W::Primal& pr = w.pr;
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const bool visc = phys_viscous(pp);
  const PhysConst<T> pc = phys_const<T>(pp);
  const GenRef& RF = *a.ref;
  const int FS = a.fs;
  for (int k = blockIdx.x; k < j.Eim; k += gridDim.x) {
    const int e = j.imp_idx[k];
    const double* gs = a.geo_sol + (size_t)a.goff[e] * 10;
    __syncthreads();  // the previous element's buffers are free
    for (int i = tid; i < N * N; i += NT) w.M[i / N][i % N] = T(RF.M[N][i / N][i % N]);
    if (tid < N) {
      w.lm[tid] = T(RF.lm[N][tid]);
      w.lp[tid] = T(RF.lp[N][tid]);
      w.dgL[tid] = T(RF.dgL[N][tid]);
      w.dgR[tid] = T(RF.dgR[N][tid]);
    }
    if (tid < nf) w.wq[tid] = T(RF.w[N][tid % N] * RF.w[N][tid / N]);
    if (tid < 6) {
      w.kf[tid] = a.kind[6 * e + tid];
      w.tr[tid] = a.tr_of[6 * e + tid];
    }
    if (tid < 5) w.uinf[tid] = T(a.uinf[tid]);
    for (int i = tid; i < ns; i += NT) {
      w.iJ[i] = T(gs[i * 10]);
      w.ciJ[i] = T(j.a_dt * gs[i * 10]);
#pragma unroll
      for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) w.Sm[i][r][c] = T(gs[i * 10 + 1 + 3 * r + c]);
    }
    for (int jj = tid; jj < 6 * nf; jj += NT) {
      const double* G = a.geo_face + ((size_t)(6 * e + jj / nf) * FS + jj % nf) * 4;
      pr.fJ[jj] = T(G[0]);
      pr.fnr[jj][0] = T(G[1]);
      pr.fnr[jj][1] = T(G[2]);
      pr.fnr[jj][2] = T(G[3]);
      w.RU[jj] = T(0);
    }
    const double* Ue = a.U + a.uoff[e];
    for (int i = tid; i < nA; i += NT) pr.U[i / HNV][i % HNV] = T(Ue[i]);
    __syncthreads();
    for (int it = tid; it < 6 * nf * HNV; it += NT) {
      const int f = it / (nf * HNV), m = (it / HNV) % nf, v = it % HNV, r = f >> 1;
      const T* l = (f & 1) ? w.lp : w.lm;
      T s = T(0);
#pragma unroll
      for (int c = 0; c < N; ++c) s += l[c] * pr.U[hline(r, m, c, N)][v];
      pr.Uf[f * nf + m][v] = s;
      const int t = w.tr[f];
      if (t >= 0) {
        pr.ub[f * nf + m][v] = T(a.uhat[(size_t)FR_IDX(a.fnode[(6 * e + f) * FS + m], a.npts, 10) * HNV + v]);
        pr.un[f * nf + m][v] = s;
      } else {  // interface face: the explicit neighbour's state
        const int nb = (int)FR_IDX(a.nbr[6 * e + f], a.E, 11), fn = (int)FR_IDX(a.nbr_face[6 * e + f], 6, 12);
        const T un = T(a.Uf_all[((size_t)(6 * nb + fn) * FS + m) * HNV + v]);
        pr.un[f * nf + m][v] = un;
        pr.ub[f * nf + m][v] = un;
      }
    }
    __syncthreads();
    if (visc) {
      for (int it = tid; it < ns * HNV; it += NT) {
        const int i = it / HNV, v = it % HNV;
        T Q[3];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          const int ar = hcoord(i, r, N), m = hfacept(i, r, N);
          T s = w.dgL[ar] * pr.ub[(2 * r) * nf + m][v] + w.dgR[ar] * pr.ub[(2 * r + 1) * nf + m][v];
#pragma unroll
          for (int c = 0; c < N; ++c) s += w.M[ar][c] * pr.U[hline(r, m, c, N)][v];
          Q[r] = s;
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) pr.q[i][c][v] = w.iJ[i] * (w.Sm[i][0][c] * Q[0] + w.Sm[i][1][c] * Q[1] + w.Sm[i][2][c] * Q[2]);
      }
      __syncthreads();
      for (int it = tid; it < 6 * nf * 3 * HNV; it += NT) {
        const int f = it / (nf * 3 * HNV), m = (it / (3 * HNV)) % nf, c2 = (it / HNV) % 3, v = it % HNV, r = f >> 1;
        const T* l = (f & 1) ? w.lp : w.lm;
        T s = T(0);
#pragma unroll
        for (int c = 0; c < N; ++c) s += l[c] * pr.q[hline(r, m, c, N)][c2][v];
        pr.qf[f * nf + m][c2][v] = s;
      }
    } else {
      for (int i = tid; i < ns * 3 * HNV; i += NT) (&pr.q[0][0][0])[i] = T(0);
      for (int i = tid; i < 6 * nf * 3 * HNV; i += NT) (&pr.qf[0][0][0])[i] = T(0);
    }
    __syncthreads();
    // ---- pointwise Jacobians (dual numbers)
    // volume: state and gradient seeds in separate whole warps
    constexpr int NI = (ns * HNV + 31) / 32 * 32, FI = (6 * nf * HNV + 31) / 32 * 32;
    for (int it = tid; it < 2 * NI; it += NT) {
      const bool isq = it >= NI;
      const int idx = isq ? it - NI : it;
      if (idx >= ns * HNV) continue;
      const int i = idx / HNV, vp = idx % HNV;
      if (!isq) {
        DT u[HNV], qd[3][HNV], F[3][HNV];
#pragma unroll
        for (int v = 0; v < HNV; ++v) {
          u[v] = DT(pr.U[i][v], v == vp ? T(1) : T(0));
#pragma unroll
          for (int c = 0; c < 3; ++c) qd[c][v] = DT(pr.q[i][c][v]);
        }
        NS3::conv<DT, T>(pc, u, F);
        if (visc) {
          DT Fv[3][HNV];
          NS3::visc<DT, T>(pc, u, qd, Fv);
#pragma unroll
          for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int v = 0; v < HNV; ++v) F[c][v] = F[c][v] - Fv[c][v];
        }
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
          for (int v = 0; v < HNV; ++v)
            J.KU[i][r][v][vp] = w.Sm[i][r][0] * F[0][v].d + w.Sm[i][r][1] * F[1][v].d + w.Sm[i][r][2] * F[2][v].d;
      } else {  // the viscous flux is linear in the gradient: its value at a unit gradient
        T acc[3][3][HNV];
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
          for (int r2 = 0; r2 < 3; ++r2)
#pragma unroll
            for (int v = 0; v < HNV; ++v) acc[r][r2][v] = T(0);
        if (visc) {
          T u[HNV], qe[3][HNV], F[3][HNV];
#pragma unroll
          for (int v = 0; v < HNV; ++v) u[v] = pr.U[i][v];
#pragma unroll
          for (int c2 = 0; c2 < 3; ++c2) {
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
              for (int v = 0; v < HNV; ++v) qe[c][v] = (c == c2 && v == vp) ? T(1) : T(0);
            NS3::visc<T, T>(pc, u, qe, F);
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
              for (int v = 0; v < HNV; ++v) {
                const T dFr = -(w.Sm[i][r][0] * F[0][v] + w.Sm[i][r][1] * F[1][v] + w.Sm[i][r][2] * F[2][v]);
#pragma unroll
                for (int r2 = 0; r2 < 3; ++r2) acc[r][r2][v] += dFr * w.iJ[i] * w.Sm[i][r2][c2];
              }
          }
        }
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
          for (int r2 = 0; r2 < 3; ++r2)
#pragma unroll
            for (int v = 0; v < HNV; ++v) J.KQ[i][r][r2][v][vp] = acc[r][r2][v];
      }
    }
    // face: 0 the trace (dual numbers), 1 the face state (traced faces J_f s 1, interface faces by dual
    // numbers), 2.. the gradient (the viscous flux at a unit gradient)
    for (int it = tid; it < 5 * FI; it += NT) {
      const int grp = it / FI, idx = it % FI;
      if (idx >= 6 * nf * HNV) continue;
      const int jj = idx / HNV, vp = idx % HNV, f = jj / nf;
      const int kf = w.kf[f];
      const bool traced = w.tr[f] >= 0;
      const T nr[3] = {pr.fnr[jj][0], pr.fnr[jj][1], pr.fnr[jj][2]}, Jf = pr.fJ[jj];
      T d[HNV], dr[HNV];
#pragma unroll
      for (int v = 0; v < HNV; ++v) d[v] = dr[v] = T(0);
      if (grp >= 2) {
        if (visc) {
          T u[HNV], qe[3][HNV], F[3][HNV];
#pragma unroll
          for (int v = 0; v < HNV; ++v) {
            u[v] = traced ? pr.ub[jj][v] : pr.Uf[jj][v];
#pragma unroll
            for (int c = 0; c < 3; ++c) qe[c][v] = (grp == 2 + c && v == vp) ? T(1) : T(0);
          }
          // faces without a trace between solved elements average both sides' viscous fluxes
          const T Ja = (!traced && (kf == FK_FR || kf == FK_FAR)) ? T(0.5) * Jf : Jf;
          NS3::visc<T, T>(pc, u, qe, F);
#pragma unroll
          for (int v = 0; v < HNV; ++v) d[v] = -Ja * (nr[0] * F[0][v] + nr[1] * F[1][v] + nr[2] * F[2][v]);
        }
      } else if (grp == 1 && traced) {
        const T s = Jf * NS3::stab<T, T>(pc, pr.ub[jj], nr);
#pragma unroll
        for (int v = 0; v < HNV; ++v) d[v] = v == vp ? s : T(0);
        if (kf == FK_FAR && vp == 0) w.RU[jj] = s;
      } else if (grp == 1 || traced) {
        DT uf[HNV], ub[HNV], un[HNV], qf[3][HNV], qn[3][HNV], Fn[HNV], row[HNV];
#pragma unroll
        for (int v = 0; v < HNV; ++v) {
          uf[v] = DT(pr.Uf[jj][v], (grp == 1 && v == vp) ? T(1) : T(0));
          ub[v] = DT(pr.ub[jj][v], (grp == 0 && v == vp) ? T(1) : T(0));
          un[v] = DT(pr.un[jj][v]);
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            qf[c][v] = DT(pr.qf[jj][c][v]);
            qn[c][v] = DT(T(0));
          }
        }
        hface_flux<DT, T>(pc, visc, kf, traced, true, uf, ub, qf, un, qn, Jf, nr, w.uinf, Fn, row);
#pragma unroll
        for (int v = 0; v < HNV; ++v) {
          d[v] = Fn[v].d;
          dr[v] = row[v].d;
        }
      }
#pragma unroll
      for (int v = 0; v < HNV; ++v) {
        if (grp == 0) {
          J.GH[jj][v][vp] = d[v];
          J.RH[jj][v][vp] = dr[v];
        } else if (grp == 1) {
          J.GU[jj][v][vp] = d[v];
        } else {
          J.GQ[jj][grp - 2][v][vp] = d[v];
        }
      }
    }
    __syncthreads();  // the primal arrays give way to the column buffers
    // ---- columns, one seed point per warp (column-major blocks: one contiguous run per column)
    T* AT = reinterpret_cast<T*>(j.A) + j.offA[k];
    T* BT = reinterpret_cast<T*>(j.B) + j.offB[k];
    T* CT = reinterpret_cast<T*>(j.C) + j.offB[k];
    T* DTm = reinterpret_cast<T*>(j.D) + j.offD[k];
    // trace unknowns of faces without a trace: zero columns of B and D
    for (int f = 0; f < 6; ++f) {
      if (w.tr[f] >= 0) continue;
      for (int it = tid; it < nf * HNV * (nA + nT); it += NT) {
        const int col = f * nf * HNV + it / (nA + nT), rr = it % (nA + nT);
        if (rr < nA)
          BT[(size_t)col * nA + rr] = T(0);
        else
          DTm[(size_t)col * nT + rr - nA] = T(0);
      }
    }
    typename W::Col& cw = w.col[wp];
    for (int sp = wp; sp < ns + 6 * nf; sp += NW) {
      const bool vol = sp < ns;
      const int f0 = vol ? -1 : (sp - ns) / nf, m0 = vol ? 0 : (sp - ns) % nf;
      if (!vol && w.tr[f0] < 0) continue;
      const int r0 = vol ? -1 : f0 >> 1;
      // seed coordinates; along the normal of a trace seed none (-1): its line runs there
      const int sx = vol ? hcoord(sp, 0, N) : (r0 == 0 ? -1 : m0 % N);
      const int sy = vol ? hcoord(sp, 1, N) : (r0 == 1 ? -1 : (r0 == 0 ? m0 % N : m0 / N));
      const int sz = vol ? hcoord(sp, 2, N) : (r0 == 2 ? -1 : m0 / N);
      const T* dg = (f0 & 1) ? w.dgR : w.dgL;  // a trace seed's weights along its line (f0 >= 0)
      auto sc = [&](int r) { return r == 0 ? sx : (r == 1 ? sy : sz); };
      // reference-gradient tangent along axis r at coordinate s of the seed's line along r
      auto line_dq = [&](int r, int s) -> T { return vol ? w.M[s][sc(r)] : dg[s]; };
      // the lines through face point (i, j) of axis r along its two tangential axes
      auto match = [&](int r, int i, int jx, bool& A, bool& B) -> bool {
        A = i == (r == 0 ? sy : sx);
        B = jx == (r == 2 ? sy : sz);
        return r == r0 ? (A && B) : (A || B);
      };
      // physical gradient tangents on the seed's lines (line r: the points that vary along r)
      for (int it = lane; it < 9 * N; it += 32) {
        const int r = it / (3 * N), s = (it / 3) % N, c = it % 3;
        if (!vol && r != r0) continue;
        const int m = vol ? hfacept(sp, r, N) : m0, pt = hline(r, m, s, N);
        T d = line_dq(r, s) * w.Sm[pt][r][c];
        if (vol && s == sc(r)) {
#pragma unroll
          for (int r2 = 0; r2 < 3; ++r2)
            if (r2 != r) d += w.M[sc(r2)][sc(r2)] * w.Sm[pt][r2][c];
        }
        cw.DQ[r][s][c] = w.iJ[pt] * d;
      }
      if (vol) {  // flux tangents at the seed point
        for (int it = lane; it < 3 * HNV; it += 32) {
          const int r = it / HNV, v = it % HNV;
#pragma unroll
          for (int x = 0; x < HNV; ++x) {
            T o = J.KU[sp][r][v][x];
#pragma unroll
            for (int r2 = 0; r2 < 3; ++r2) o += J.KQ[sp][r][r2][v][x] * w.M[sc(r2)][sc(r2)];
            cw.SD[r][v][x] = o;
          }
        }
      }
      __syncwarp();
      // gradient tangents at the active face points: slot a (first tangential coordinate that of the
      // seed) at the second coordinate, slot N + b (second that of the seed) at the first
      for (int it = lane; it < 6 * 2 * N * 3; it += 32) {
        const int f = it / (6 * N), sl = (it / 3) % (2 * N), c = it % 3, r = f >> 1;
        const int t0 = r == 0 ? 1 : 0, t1 = r == 2 ? 1 : 2;
        const int i = sl < N ? sc(t0) : sl - N, jx = sl < N ? sl : sc(t1);
        if (i < 0 || jx < 0) continue;
        bool A, B;
        if (!match(r, i, jx, A, B)) continue;
        const T* l = (f & 1) ? w.lp : w.lm;
        T s = T(0);
        if (A && B) {  // the normal line is the seed's own
#pragma unroll
          for (int c1 = 0; c1 < N; ++c1) s += l[c1] * cw.DQ[r][c1][c];
        } else {  // it meets the seed's line along t1 (A) or t0 (B) in one point
          s = l[sc(r)] * (A ? cw.DQ[t1][jx][c] : cw.DQ[t0][i][c]);
        }
        cw.qf[f][sl][c] = s;
      }
      // line sums
      for (int it = lane; it < 3 * N * HNV; it += 32) {
        const int r = it / (N * HNV), i = (it / HNV) % N, v = it % HNV;
        if (!vol && r != r0) continue;
        const int m = vol ? hfacept(sp, r, N) : m0;
        T o[HNV];
#pragma unroll
        for (int x = 0; x < HNV; ++x) o[x] = T(0);
#pragma unroll
        for (int s = 0; s < N; ++s) {
          if (vol && s == sc(r)) {
#pragma unroll
            for (int x = 0; x < HNV; ++x) o[x] += w.M[i][s] * cw.SD[r][v][x];
          } else {
            const T cf = w.M[i][s] * line_dq(r, s);
            const T* kq = &J.KQ[hline(r, m, s, N)][r][r][v][0];
#pragma unroll
            for (int x = 0; x < HNV; ++x) o[x] += cf * kq[x];
          }
        }
#pragma unroll
        for (int x = 0; x < HNV; ++x) cw.RC[r][i][v][x] = o[x];
      }
      __syncwarp();
      // face flux tangents at the active points
      for (int it = lane; it < 6 * 2 * N * HNV; it += 32) {
        const int f = it / (2 * N * HNV), sl = (it / HNV) % (2 * N), v = it % HNV, r = f >> 1;
        const int t0 = r == 0 ? 1 : 0, t1 = r == 2 ? 1 : 2;
        const int i = sl < N ? sc(t0) : sl - N, jx = sl < N ? sl : sc(t1);
        if (i < 0 || jx < 0) continue;
        bool A, B;
        if (!match(r, i, jx, A, B)) continue;
        const int jj = f * nf + i + N * jx;
        const T q0 = cw.qf[f][sl][0], q1 = cw.qf[f][sl][1], q2 = cw.qf[f][sl][2];
        T o[HNV];
#pragma unroll
        for (int x = 0; x < HNV; ++x)
          o[x] = J.GQ[jj][0][v][x] * q0 + J.GQ[jj][1][v][x] * q1 + J.GQ[jj][2][v][x] * q2;
        if (vol && A && B) {  // the face state on the seed's own normal line
          const T du = ((f & 1) ? w.lp : w.lm)[sc(r)];
#pragma unroll
          for (int x = 0; x < HNV; ++x) o[x] += J.GU[jj][v][x] * du;
        }
        if (f == f0 && A && B) {
#pragma unroll
          for (int x = 0; x < HNV; ++x) o[x] += J.GH[jj][v][x];
        }
#pragma unroll
        for (int x = 0; x < HNV; ++x) cw.FN[f][sl][v][x] = o[x];
      }
      __syncwarp();
      const int col = vol ? sp * HNV : (f0 * nf + m0) * HNV;
      T* top = (vol ? AT : BT) + (size_t)col * nA;
      T* bot = (vol ? CT : DTm) + (size_t)col * nT;
      // A / B columns: a dt / J times the divergence tangent (plus the identity of A)
      for (int it = lane; it < nA; it += 32) {
        const int pt = it / HNV, v = it % HNV;
        T o[HNV];
#pragma unroll
        for (int x = 0; x < HNV; ++x) o[x] = T(0);
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          const int t0 = r == 0 ? 1 : 0, t1 = r == 2 ? 1 : 2;
          const int ar = hcoord(pt, r, N), i = hcoord(pt, t0, N), jx = hcoord(pt, t1, N);
          bool A, B;
          if (!match(r, i, jx, A, B)) continue;
          if (A && B) {
#pragma unroll
            for (int x = 0; x < HNV; ++x) o[x] += cw.RC[r][ar][v][x];
          } else {  // (sc(r) >= 0: a trace seed along r has A and B together)
            const int tl = A ? t1 : t0, s = A ? jx : i;
            const T cf = w.M[ar][sc(r)] * line_dq(tl, s);
            const T* kq = &J.KQ[hline(r, i + N * jx, sc(r), N)][r][tl][v][0];
#pragma unroll
            for (int x = 0; x < HNV; ++x) o[x] += cf * kq[x];
          }
          const int sl = A ? jx : N + i;
          const T gl = -w.dgL[ar], gr = w.dgR[ar];
          const T* fl = &cw.FN[2 * r][sl][v][0];
          const T* fr = &cw.FN[2 * r + 1][sl][v][0];
#pragma unroll
          for (int x = 0; x < HNV; ++x) o[x] += gl * fl[x] + gr * fr[x];
        }
        const T cj = w.ciJ[pt];
#pragma unroll
        for (int x = 0; x < HNV; ++x) {
          T y = cj * o[x];
          if (vol && it == col + x) y += T(1);
          top[(size_t)x * nA + it] = y;
        }
      }
      // C / D columns: w_q times the trace row's tangent (walls: momentum rows of the trace alone;
      // far field: J_f s (u_f - u^) and the trace's own part)
      for (int it = lane; it < nT; it += 32) {
        const int jj = it / HNV, v = it % HNV, f = jj / nf, m = jj % nf, r = f >> 1, kf = w.kf[f];
        T o[HNV];
#pragma unroll
        for (int x = 0; x < HNV; ++x) o[x] = T(0);
        bool A, B;
        if (w.tr[f] >= 0 && match(r, m % N, m / N, A, B)) {
          const bool wall = kf == FK_WALL && v != 0 && v != HNV - 1;
          if (!wall && kf != FK_FAR) {
            const T* fn = &cw.FN[f][A ? m / N : N + m % N][v][0];
#pragma unroll
            for (int x = 0; x < HNV; ++x) o[x] = fn[x];
          } else {
            if (f == f0 && m == m0) {
#pragma unroll
              for (int x = 0; x < HNV; ++x) o[x] = J.RH[jj][v][x];
            }
            if (kf == FK_FAR && vol && A && B) {
              const T du = w.RU[jj] * ((f & 1) ? w.lp : w.lm)[sc(r)];
#pragma unroll
              for (int x = 0; x < HNV; ++x)
                if (x == v) o[x] += du;
            }
          }
          const T wm = w.wq[m];
#pragma unroll
          for (int x = 0; x < HNV; ++x) o[x] *= wm;
        }
#pragma unroll
        for (int x = 0; x < HNV; ++x) bot[(size_t)x * nT + it] = o[x];
      }
      __syncwarp();
    }
  }
}

int hex_jacobian_grid(int prec_bytes) {
  (void)prec_bytes;
  int dev = 0, nsm = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  return nsm;
}

size_t hex_jacobian_scratch_bytes(int prec_bytes, int grid) {
  return prec_bytes == 8 ? (size_t)grid * sizeof(HJac<double, HN>) : 0;  // FP32 keeps them in shared memory
}

template <typename T, int N>
static cudaError_t hex_jac_launch(GenCtx* g, const GArgs& a, const JArgs& j) {
  const size_t smem = hex_jac_smem<T, N>();
  auto kern = k_hex_jacobian<T, N>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  (count_launch(), kern<<<g->jgrid, 32 * HJWork<T, N>::NW, smem, g->st>>>(g->pp, a, j));
  return cudaGetLastError();
}
cudaError_t hex_jacobian(GenCtx* g, const GArgs& a, const JArgs& j) {
  if (j.Eim == 0) return cudaSuccess;
  const bool f64 = g->pb == 8;
  switch (g->h_deg.empty() ? 0 : g->h_deg[0]) {  // hexahedral meshes carry one degree
    case 2: return f64 ? hex_jac_launch<double, 2>(g, a, j) : hex_jac_launch<float, 2>(g, a, j);
    case 3: return f64 ? hex_jac_launch<double, 3>(g, a, j) : hex_jac_launch<float, 3>(g, a, j);
    case 4: return f64 ? hex_jac_launch<double, 4>(g, a, j) : hex_jac_launch<float, 4>(g, a, j);
    default: return cudaErrorInvalidValue;
  }
}

// ------------------------------------------------------------------------ geometry (host)
void hex_geometry(const double* verts, int E, const int* deg, const long long* goff, double* gsol, double* gface,
                  double* xyz) {
  for (int e = 0; e < E; ++e) {
    const int n = deg[e];
    double x[HN], wg[HN];
    gauss_legendre_nodes(n, x, wg);
    const double* V = verts + (size_t)e * 24;
    auto map = [&](const double r[3], double X[3], double D[3][3]) {  // D[k] = dx/dxi_k
      for (int c = 0; c < 3; ++c) {
        X[c] = 0.0;
        D[0][c] = D[1][c] = D[2][c] = 0.0;
      }
      for (int k = 0; k < 8; ++k) {
        const double s[3] = {(k & 1) ? 1.0 : -1.0, (k & 2) ? 1.0 : -1.0, (k & 4) ? 1.0 : -1.0};
        const double f0 = 1 + s[0] * r[0], f1 = 1 + s[1] * r[1], f2 = 1 + s[2] * r[2];
        const double N = 0.125 * f0 * f1 * f2;
        const double dN[3] = {0.125 * s[0] * f1 * f2, 0.125 * s[1] * f0 * f2, 0.125 * s[2] * f0 * f1};
        for (int c = 0; c < 3; ++c) {
          X[c] += N * V[3 * k + c];
          for (int d = 0; d < 3; ++d) D[d][c] += dN[d] * V[3 * k + c];
        }
      }
    };
    auto cross = [](const double* u, const double* v, double* o) {
      o[0] = u[1] * v[2] - u[2] * v[1];
      o[1] = u[2] * v[0] - u[0] * v[2];
      o[2] = u[0] * v[1] - u[1] * v[0];
    };
    auto adj = [&](double D[3][3], double S[3][3]) {  // S[r] = x_{xi_s} x x_{xi_t}, (r, s, t) cyclic
      cross(D[1], D[2], S[0]);
      cross(D[2], D[0], S[1]);
      cross(D[0], D[1], S[2]);
      return D[0][0] * S[0][0] + D[0][1] * S[0][1] + D[0][2] * S[0][2];
    };
    for (int c3 = 0; c3 < n; ++c3)
      for (int b = 0; b < n; ++b)
        for (int a2 = 0; a2 < n; ++a2) {
          const size_t pt = (size_t)goff[e] + a2 + n * b + n * n * c3;
          const double r[3] = {x[a2], x[b], x[c3]};
          double X[3], D[3][3], S[3][3];
          map(r, X, D);
          const double J = adj(D, S);
          double* G = gsol + 10 * pt;
          G[0] = 1.0 / J;
          for (int rr = 0; rr < 3; ++rr)
            for (int cc = 0; cc < 3; ++cc) G[1 + 3 * rr + cc] = S[rr][cc];
          for (int cc = 0; cc < 3; ++cc) xyz[3 * pt + cc] = X[cc];
        }
    for (int f = 0; f < 6; ++f) {
      const int rax = f >> 1;
      const double sg = (f & 1) ? 1.0 : -1.0;
      const int t0 = rax == 0 ? 1 : 0, t1 = rax == 2 ? 1 : 2;  // lower and higher tangential axes
      for (int jj = 0; jj < n; ++jj)
        for (int ii = 0; ii < n; ++ii) {
          double r[3];
          r[rax] = sg;
          r[t0] = x[ii];
          r[t1] = x[jj];
          double X[3], D[3][3], S[3][3];
          map(r, X, D);
          adj(D, S);
          const double N[3] = {sg * S[rax][0], sg * S[rax][1], sg * S[rax][2]};
          const double Jf = sqrt(N[0] * N[0] + N[1] * N[1] + N[2] * N[2]);
          double* G = gface + 4 * ((size_t)(6 * e + f) * HEX_FS + ii + n * jj);
          G[0] = Jf;
          G[1] = N[0] / Jf;
          G[2] = N[1] / Jf;
          G[3] = N[2] / Jf;
        }
    }
  }
}

}  // namespace gen
}  // namespace hfr

#include "hfr_checked_unit.inc"
