// FR / hybridized-FR residual kernels (Pereira & Vermeire, arXiv 2401.16632, Sec. 2:
// eqs. freq1, hfrriemann, hfr1; transmission conditions eqs. 5treerf, hfr2; IMEX
// interface eq. hfrimex).
//
// A CTA takes EPB elements and walks each phase's items (solution points, face points, or their
// single values) over all of them, so that the items fill whole warps: the residual is FP64 and
// bound by the FP64 pipe, where a warp costs the same with 9 live lanes as with 32 (one element per
// warp left 28 % of the lanes live at p = 2, 50 % at p = 3, 56 % at p = 5).  Linear operations go by
// single values (one chain per thread); face fluxes are formed as normal components only.  On meshes
// with explicit elements the neighbours' face states and gradients are formed by two passes first
// (MODE_UF, MODE_QF); the second also keeps the gradients of the solution points, and the residual
// pass (MODE_RESQ) starts from both instead of forming them again.
// Measured (one residual): 203 x 177 elements, p = 5, an implicit band: 2.19 -> 1.01 ms; 256 x 256,
// p = 4: 1.51 -> 1.13 ms; 64 x 64, p = 3: 95 -> 54 us; 61 x 47, p = 2 with a band: 105 -> 49 us.
//
// The element computation is a template on the scalar type S: S = double gives the residual,
// S = Dual<double> the residual and its exact directional derivative (refinement residuals of the
// local solves).
#include "hfr_internal.h"

namespace hfr {

template <int P, int PHYS, typename S>
struct ElemWork {
  static constexpr int N = P + 1, NS = N * N, NV = Phys<PHYS>::NV, NF = 4 * N;
  S U[NS][NV];
  S Uf[NF][NV];
  S ub[NF][NV];
  S q[NS][2][NV];
  S qf[NF][2][NV];
  S Ft[NS][2][NV];
  S Fn[NF][NV];
};

template <typename S> __device__ __forceinline__ S mk(double v, double d);
template <> __device__ __forceinline__ double mk<double>(double v, double) { return v; }
template <> __device__ __forceinline__ Dual<double> mk<Dual<double>>(double v, double d) { return Dual<double>(v, d); }
__device__ __forceinline__ double tangent(double) { return 0.0; }
__device__ __forceinline__ double tangent(Dual<double> a) { return a.d; }

// Modes of the element kernel: face states; face gradients (and the solution points'); the residual
// from the states alone; the residual from stored face states and gradients (FP64 values only).
enum { MODE_UF = 0, MODE_QF = 1, MODE_RES = 2, MODE_RESQ = 3 };

// shared memory of one element in each mode
template <int P, int PHYS, typename S, int MODE>
constexpr size_t elem_smem() {
  using W = ElemWork<P, PHYS, S>;
  return MODE == MODE_RESQ ? sizeof(S) * W::NV * (2 * W::NS + W::NF)  // Ft, Fn
         : MODE == MODE_RES ? sizeof(W)
                            : sizeof(S) * W::NV * (W::NS + 2 * W::NF + (MODE == MODE_QF ? 2 * W::NS : 0));
}

template <int P, int PHYS, typename S, int MODE, int EPB, int NT>
__global__ void __launch_bounds__(NT) k_element(const __grid_constant__ RefOps ref,
                                                const __grid_constant__ PhysParams pp,
                                                const __grid_constant__ ResArgs a) {
  using W = ElemWork<P, PHYS, S>;
  using PH = Phys<PHYS>;
  constexpr int N = W::N, NS = W::NS, NV = W::NV, NF = W::NF;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  S* base = reinterpret_cast<S*>(smem_raw);
  // per-phase arrays over the CTA's elements, [EPB][..][NV]
  S* sU = base;                                          // NS       (all but RESQ)
  S* sUf = sU + EPB * NS * NV;                           // NF
  S* sub = sUf + EPB * NF * NV;                          // NF
  S* sq = sub + EPB * NF * NV;                           // NS x 2   (QF, RES)
  S* sqf = sq + EPB * NS * 2 * NV;                       // NF x 2   (RES)
  S* sFt = MODE == MODE_RESQ ? base : sqf + EPB * NF * 2 * NV;  // NS x 2 (RES, RESQ)
  S* sFn = sFt + EPB * NS * 2 * NV;                      // NF       (RES, RESQ)
  const int tid = threadIdx.x;
  const int e0 = blockIdx.x * EPB;
  const int ne = min(EPB, a.E - e0);
  const bool viscous = phys_viscous(pp);
  const PhysConst<double> pc = phys_const<double>(pp);
  const double* gs = a.geo_sol + (size_t)e0 * NS * 5;
  const double* gf = a.geo_face + (size_t)e0 * NF * 3;

  if constexpr (MODE != MODE_RESQ) {
    // 1. state
    for (int i = tid; i < ne * NS * NV; i += NT) {
      const size_t ix = (size_t)e0 * NS * NV + i;
      sU[i] = mk<S>(a.U[ix], a.dU ? a.dU[ix] : 0.0);
    }
    __syncthreads();
    // 2. face states and common solution
    for (int it = tid; it < ne * NF * NV; it += NT) {
      const int v = it % NV, j = (it / NV) % NF, el = it / (NV * NF), f = j / N, m = j % N, r = f >> 1, e = e0 + el;
      S uf;
      if (MODE == MODE_QF) {
        uf = S(a.Uf_all[(size_t)e0 * NF * NV + it]);
      } else {
        const double* l = (f & 1) ? ref.lp : ref.lm;
        uf = S(0.0);
#pragma unroll
        for (int c = 0; c < N; ++c) uf = uf + l[c] * sU[(el * NS + line_pt<N>(r, m, c)) * NV + v];
      }
      if (MODE == MODE_UF) {
        a.Uf_out[(size_t)e0 * NF * NV + it] = dval(uf);
        continue;
      }
      sUf[it] = uf;
      const int kf = a.kind[e * 4 + f];
      if (kf == FK_TRACE) {
        const int t = (int)FR_IDX(a.tr_of[e * 4 + f], a.ntrace, 20);
        const size_t ix = ((size_t)t * N + m) * NV + v;
        sub[it] = mk<S>(a.uhat[ix], a.duhat ? a.duhat[ix] : 0.0);
      } else {
        const int en = (int)FR_IDX(a.nbr[e * 4 + f], a.E, 21), fn = (int)FR_IDX(a.nbr_face[e * 4 + f], 4, 22);
        const S un = S(a.Uf_all[((size_t)en * NF + fn * N + m) * NV + v]);
        // IMEX interface: the explicit side's value
        sub[it] = kf == FK_FR ? 0.5 * (uf + un) : (a.implicit[e] ? un : uf);
      }
    }
    if constexpr (MODE == MODE_UF) return;
    __syncthreads();
    // 3. corrected gradient at the solution points
    if (viscous) {
      for (int it = tid; it < ne * NS * NV; it += NT) {
        const int v = it % NV, i = (it / NV) % NS, el = it / (NV * NS), ai = i % N, bi = i / N;
        const double* G = gs + (size_t)(el * NS + i) * 5;
        const S* U = sU + el * NS * NV + v;
        const S* ub = sub + el * NF * NV + v;
        S q0 = ref.dgL[ai] * ub[(0 * N + bi) * NV] + ref.dgR[ai] * ub[(1 * N + bi) * NV];
        S q1 = ref.dgL[bi] * ub[(2 * N + ai) * NV] + ref.dgR[bi] * ub[(3 * N + ai) * NV];
#pragma unroll
        for (int c = 0; c < N; ++c) {
          q0 = q0 + ref.M[ai][c] * U[(c + N * bi) * NV];
          q1 = q1 + ref.M[bi][c] * U[(ai + N * c) * NV];
        }
        const S qx = G[0] * (G[1] * q0 + G[3] * q1), qy = G[0] * (G[2] * q0 + G[4] * q1);
        S* q = sq + (size_t)(el * NS + i) * 2 * NV + v;
        q[0] = qx;
        q[NV] = qy;
        if (MODE == MODE_QF) {
          double* o = a.q_out + ((size_t)(e0 + el) * NS + i) * 2 * NV + v;
          o[0] = dval(qx);
          o[NV] = dval(qy);
        }
      }
      __syncthreads();
      // 4. gradient at the flux points
      for (int it = tid; it < ne * NF * 2 * NV; it += NT) {
        const int cv = it % (2 * NV), j = (it / (2 * NV)) % NF, el = it / (2 * NV * NF), f = j / N, m = j % N, r = f >> 1;
        const double* l = (f & 1) ? ref.lp : ref.lm;
        S s = S(0.0);
#pragma unroll
        for (int c = 0; c < N; ++c) s = s + l[c] * sq[(el * NS + line_pt<N>(r, m, c)) * 2 * NV + cv];
        if (MODE == MODE_QF)
          a.qf_out[(size_t)e0 * NF * 2 * NV + it] = dval(s);
        else
          sqf[it] = s;
      }
    } else if (MODE == MODE_QF) {
      for (int j = tid; j < ne * NF * 2 * NV; j += NT) a.qf_out[(size_t)e0 * NF * 2 * NV + j] = 0.0;
    }
  }
  if constexpr (MODE == MODE_RES || MODE == MODE_RESQ) {
  // 5. transformed flux at the solution points
  for (int it = tid; it < ne * NS; it += NT) {
    const double* G = gs + (size_t)it * 5;
    S u[NV], q[2][NV], F[2][NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      if constexpr (MODE == MODE_RESQ)
        u[v] = S(a.U[((size_t)e0 * NS + it) * NV + v]);
      else
        u[v] = sU[it * NV + v];
    }
    PH::template conv<S, double>(pc, u, F);
    if (viscous) {
      S Fv[2][NV];
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          if constexpr (MODE == MODE_RESQ)
            q[c][v] = S(a.q_out[(((size_t)e0 * NS + it) * 2 + c) * NV + v]);
          else
            q[c][v] = sq[(it * 2 + c) * NV + v];
        }
      PH::template visc<S, double>(pc, u, q, Fv);
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int v = 0; v < NV; ++v) F[c][v] = F[c][v] - Fv[c][v];
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      sFt[(it * 2 + 0) * NV + v] = G[1] * F[0][v] + G[2] * F[1][v];
      sFt[(it * 2 + 1) * NV + v] = G[3] * F[0][v] + G[4] * F[1][v];
    }
  }
  if constexpr (MODE == MODE_RES) __syncthreads();  // the flux points' gradients
  // 6. common normal flux Fn = J_f F^.n at every flux point
  for (int it = tid; it < ne * NF; it += NT) {
    const int j = it % NF, e = e0 + it / NF, f = j / N, m = j % N;
    const double* G = gf + (size_t)it * 3;
    const double Jf = G[0], n0 = G[1], n1 = G[2];
    const int kf = a.kind[e * 4 + f];
    S uf[NV], qf[2][NV], Fh[NV], wv;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      if constexpr (MODE == MODE_RESQ)
        uf[v] = S(a.Uf_all[((size_t)e0 * NF + it) * NV + v]);
      else
        uf[v] = sUf[it * NV + v];
      if (viscous) {
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          if constexpr (MODE == MODE_RESQ)
            qf[c][v] = S(a.qf_all[(((size_t)e0 * NF + it) * 2 + c) * NV + v]);
          else
            qf[c][v] = sqf[(it * 2 + c) * NV + v];
        }
      }
    }
    if (kf == FK_TRACE) {
      S ub[NV], Fv[NV];
      const size_t tx = MODE == MODE_RESQ ? ((size_t)FR_IDX(a.tr_of[e * 4 + f], a.ntrace, 20) * N + m) * NV : 0;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        if constexpr (MODE == MODE_RESQ)
          ub[v] = S(a.uhat[tx + v]);
        else
          ub[v] = sub[it * NV + v];
      }
      PH::template conv_n<S, double>(pc, ub, n0, n1, Fh, wv);
      const S s = PH::template stab_n<S, double>(pc, ub, wv);
#pragma unroll
      for (int v = 0; v < NV; ++v) Fh[v] = Fh[v] + s * (uf[v] - ub[v]);
      if (viscous) {
        PH::template visc_n<S, double>(pc, ub, qf, n0, n1, Fv);
#pragma unroll
        for (int v = 0; v < NV; ++v) Fh[v] = Fh[v] - Fv[v];
      }
    } else {
      const int en = (int)FR_IDX(a.nbr[e * 4 + f], a.E, 21), fn = (int)FR_IDX(a.nbr_face[e * 4 + f], 4, 22);
      const size_t nix = (size_t)en * NF + fn * N + m;
      S un[NV], Fb[NV], wn;
#pragma unroll
      for (int v = 0; v < NV; ++v) un[v] = S(a.Uf_all[nix * NV + v]);
      PH::template conv_n<S, double>(pc, uf, n0, n1, Fh, wv);
      PH::template conv_n<S, double>(pc, un, n0, n1, Fb, wn);
      const S lam = dmax(wv, wn);
#pragma unroll
      for (int v = 0; v < NV; ++v) Fh[v] = 0.5 * (Fh[v] + Fb[v]) + 0.5 * lam * (uf[v] - un[v]);
      if (viscous) {
        const bool im = a.implicit[e] != 0;
        S qn[2][NV], Fv[NV];
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int v = 0; v < NV; ++v) qn[c][v] = S(a.qf_all[(nix * 2 + c) * NV + v]);
        if (kf == FK_FR) {  // both sides' viscous fluxes averaged
          PH::template visc_n<S, double>(pc, uf, qf, n0, n1, Fv);
          PH::template visc_n<S, double>(pc, un, qn, n0, n1, Fb);
#pragma unroll
          for (int v = 0; v < NV; ++v) Fh[v] = Fh[v] - 0.5 * (Fv[v] + Fb[v]);
        } else {  // IMEX interface: the implicit side's
          if (im)
            PH::template visc_n<S, double>(pc, uf, qf, n0, n1, Fv);
          else
            PH::template visc_n<S, double>(pc, un, qn, n0, n1, Fv);
#pragma unroll
          for (int v = 0; v < NV; ++v) Fh[v] = Fh[v] - Fv[v];
        }
      }
    }
    // element contribution to the trace residual (zero off trace faces)
    const double wq = kf == FK_TRACE ? ref.w[m] : 0.0;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const S Fn = Jf * Fh[v];
      sFn[it * NV + v] = Fn;
      if (a.gview) {
        const size_t ix = ((size_t)e0 * NF + it) * NV + v;
        a.gview[ix] = wq * dval(Fn);
        if (a.dgview) a.dgview[ix] = wq * tangent(Fn);
      }
    }
  }
  __syncthreads();
  // 7. divergence: R = -(1/J) [sum_r M F~_r - dgL Fn_L + dgR Fn_R]
  for (int it = tid; it < ne * NS * NV; it += NT) {
    const int v = it % NV, i = (it / NV) % NS, el = it / (NV * NS), ai = i % N, bi = i / N;
    const S* Ft = sFt + el * NS * 2 * NV + v;
    const S* Fn = sFn + el * NF * NV + v;
    S d = -ref.dgL[ai] * Fn[(0 * N + bi) * NV] + ref.dgR[ai] * Fn[(1 * N + bi) * NV] -
          ref.dgL[bi] * Fn[(2 * N + ai) * NV] + ref.dgR[bi] * Fn[(3 * N + ai) * NV];
#pragma unroll
    for (int c = 0; c < N; ++c)
      d = d + ref.M[ai][c] * Ft[(c + N * bi) * 2 * NV] + ref.M[bi][c] * Ft[((ai + N * c) * 2 + 1) * NV];
    const S Rv = -gs[(size_t)(el * NS + i) * 5] * d;
    const size_t ix = (size_t)e0 * NS * NV + it;
    if (a.R) a.R[ix] = dval(Rv);
    if (a.dR) a.dR[ix] = tangent(Rv);
  }
  }
}

// trace residual: g[t] = gview(side 0) + gview(side 1)
__global__ void k_trace_assemble(const double* __restrict__ gview, const int* __restrict__ sides, int ntrace,
                                 int npf, double* __restrict__ g) {
  // npf = values per face = n * nv; element face stride = 4 * n * nv
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ntrace * npf) return;
  const int t = i / npf, k = i % npf;
  const int e0 = sides[t * 4 + 0], f0 = sides[t * 4 + 1], e1 = sides[t * 4 + 2], f1 = sides[t * 4 + 3];
  double s = gview[((size_t)e0 * 4 + f0) * npf + k];
  if (e1 >= 0) s += gview[((size_t)e1 * 4 + f1) * npf + k];
  g[i] = s;
}

// -------------------------------------------------------------------------------------------
template <int P, int PHYS, typename S, int MODE, int EPB, int NT>
static cudaError_t launch_elem_n(const RefOps& ref, const PhysParams& pp, const ResArgs& a, cudaStream_t st) {
  constexpr size_t smem = elem_smem<P, PHYS, S, MODE>() * EPB;
  static_assert(smem <= 227 * 1024, "residual workspace exceeds shared memory");
  auto kern = k_element<P, PHYS, S, MODE, EPB, NT>;
  cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  const int grid = (a.E + EPB - 1) / EPB;
  if (grid == 0) return cudaSuccess;
  (hfr::count_launch(), kern<<<grid, NT, smem, st>>>(ref, pp, a));
  return cudaGetLastError();
}
// elements per CTA: as many as fill whole warps with points (p = 2: 144 points of 160 lanes; p = 3
// and 5: all lanes; p = 4: 200 of 224), fewer where that would leave less than two CTAs per SM:
// there the passes last a few microseconds and a phase's latency counts, not its lanes (an IMEX step of
// 2867 elements, p = 2: 2.40 ms with 16 elements per CTA, 2.29 ms with 4)
template <int P, int PHYS, typename S, int MODE>
static cudaError_t launch_elem(const RefOps& ref, const PhysParams& pp, const ResArgs& a, cudaStream_t st) {
  constexpr int EPB = P <= 2 ? 16 : 8, NT = P <= 3 ? 128 : 256;
  if (a.E >= 2 * a.nsm * EPB) return launch_elem_n<P, PHYS, S, MODE, EPB, NT>(ref, pp, a, st);
  return launch_elem_n<P, PHYS, S, MODE, 4, 128>(ref, pp, a, st);
}

template <int P, int PHYS>
static cudaError_t residual_impl(const RefOps& ref, const PhysParams& pp, ResArgs a, bool need_nbr, bool jvp,
                                 cudaStream_t st) {
  cudaError_t err;
  if (need_nbr) {
    // neighbour face states and gradients (FR and interface faces); tangents of the
    // neighbour data are not propagated (explicit states are held fixed).
    ResArgs b = a;
    b.dU = nullptr;
    b.duhat = nullptr;
    if ((err = launch_elem<P, PHYS, double, MODE_UF>(ref, pp, b, st)) != cudaSuccess) return err;
    if ((err = launch_elem<P, PHYS, double, MODE_QF>(ref, pp, b, st)) != cudaSuccess) return err;
    if (!jvp) return launch_elem<P, PHYS, double, MODE_RESQ>(ref, pp, a, st);
  }
  if (jvp) return launch_elem<P, PHYS, Dual<double>, MODE_RES>(ref, pp, a, st);
  return launch_elem<P, PHYS, double, MODE_RES>(ref, pp, a, st);
}

cudaError_t launch_residual(int p, const RefOps& ref, const PhysParams& pp, const ResArgs& a, bool need_nbr, bool jvp,
                            cudaStream_t st) {
  if (pp.kind == 0) {
    switch (p) {
      case 1: return residual_impl<1, 0>(ref, pp, a, need_nbr, jvp, st);
      case 2: return residual_impl<2, 0>(ref, pp, a, need_nbr, jvp, st);
      case 3: return residual_impl<3, 0>(ref, pp, a, need_nbr, jvp, st);
    }
  } else if (pp.kind == 2) {
    switch (p) {
      case 2: return residual_impl<2, 2>(ref, pp, a, need_nbr, jvp, st);
      case 3: return residual_impl<3, 2>(ref, pp, a, need_nbr, jvp, st);
      case 4: return residual_impl<4, 2>(ref, pp, a, need_nbr, jvp, st);
    }
  } else {
    switch (p) {
      case 2: return residual_impl<2, 1>(ref, pp, a, need_nbr, jvp, st);
      case 3: return residual_impl<3, 1>(ref, pp, a, need_nbr, jvp, st);
      case 4: return residual_impl<4, 1>(ref, pp, a, need_nbr, jvp, st);
      case 5: return residual_impl<5, 1>(ref, pp, a, need_nbr, jvp, st);
    }
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_face_states(int p, const RefOps& ref, const PhysParams& pp, const ResArgs& a, cudaStream_t st) {
  if (pp.kind == 0) {
    switch (p) {
      case 1: return launch_elem<1, 0, double, MODE_UF>(ref, pp, a, st);
      case 2: return launch_elem<2, 0, double, MODE_UF>(ref, pp, a, st);
      case 3: return launch_elem<3, 0, double, MODE_UF>(ref, pp, a, st);
    }
  } else if (pp.kind == 2) {
    switch (p) {
      case 2: return launch_elem<2, 2, double, MODE_UF>(ref, pp, a, st);
      case 3: return launch_elem<3, 2, double, MODE_UF>(ref, pp, a, st);
      case 4: return launch_elem<4, 2, double, MODE_UF>(ref, pp, a, st);
    }
  } else {
    switch (p) {
      case 2: return launch_elem<2, 1, double, MODE_UF>(ref, pp, a, st);
      case 3: return launch_elem<3, 1, double, MODE_UF>(ref, pp, a, st);
      case 4: return launch_elem<4, 1, double, MODE_UF>(ref, pp, a, st);
      case 5: return launch_elem<5, 1, double, MODE_UF>(ref, pp, a, st);
    }
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_trace_assemble(const double* gview, const int* sides, int ntrace, int npf, double* g,
                                  cudaStream_t st) {
  int total = ntrace * npf;
  if (total == 0) return cudaSuccess;
  (hfr::count_launch(), k_trace_assemble<<<(total + 255) / 256, 256, 0, st>>>(gview, sides, ntrace, npf, g));
  return cudaGetLastError();
}

}  // namespace hfr

#include "hfr_checked_unit.inc"
