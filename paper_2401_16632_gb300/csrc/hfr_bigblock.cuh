// Condensation of element blocks too large for one CTA's shared memory (FP64 p = 5 quadrilaterals,
// hexahedra: nA = 320, nT = 480), as a sequence of batched kernels over all such elements:
//   1. blocked right-looking LU with partial pivoting of A in place, panel by panel of LB columns:
//      the panel (all its rows) factorised in shared memory by one CTA per element (largest |a|,
//      lowest row on ties), its row interchanges applied to the columns left and right of it and
//      the block row right of it solved with the panel's unit lower triangle (same kernel); then
//      the trailing matrix updated by the batched GEMM;
//   2-3. X = A^{-1} P [B | r]: one CTA per block of columns of one element, the block whole in shared
//      memory (permuted columns in, forward and back substitution by factor panels, X out once);
//   4. S = D - C X_B, in FP32 on the tensor cores, in FP64 by the same batched GEMM;
//   5. t = s - C x_r with FP64 accumulation (one CTA per element); x_r is the right-hand side's column
//      of step 2-3, in batches with FP32 blocks of more than XR32_MAX rows a substitution in FP64.
// The batched GEMM is a register-tiled CUDA-core kernel: 128 x 128 output tiles in FP32 (32 x 32 in
// FP64), 256 threads with 8 x 8 (2 x 2) outputs each, K staged through two shared-memory buffers 8
// at a time; arithmetic in the block precision T.  Included by hfr_condense.cu (uses UnevenArgs and DEV_ERR_*).
#pragma once

namespace hfr {
namespace big {

constexpr int BT = 256;      // threads per CTA
// LU panel width: the panel of up to 1024 rows stays in shared memory (128 KB at most)
template <typename T>
__host__ __device__ constexpr int lu_panel() {
  return sizeof(T) == 8 ? 16 : 32;
}
template <typename T>
size_t lu_panel_smem(int max_nA) {
  return (size_t)max_nA * (lu_panel<T>() + 1) * sizeof(T);
}

// element of list position li: its id, five offsets and shape (tables, or one uniform shape)
struct Elem {
  int k, nA, nT;
  long long o[5];
};
__device__ __forceinline__ Elem elem_of(const UnevenArgs& a, const int* list, int li, int uni_nA, int uni_nT) {
  Elem e;
  e.k = list ? list[li] : li;
  if (uni_nA > 0) {
    e.nA = uni_nA;
    e.nT = uni_nT;
    e.o[0] = (long long)e.k * e.nA * e.nA;
    e.o[1] = (long long)e.k * e.nA * e.nT;
    e.o[2] = (long long)e.k * e.nT * e.nT;
    e.o[3] = (long long)e.k * e.nA;
    e.o[4] = (long long)e.k * e.nT;
  } else {
#pragma unroll
    for (int q = 0; q < 5; ++q) e.o[q] = a.off[5 * (size_t)e.k + q];
    e.nA = a.shape[2 * e.k];
    e.nT = a.shape[2 * e.k + 1];
  }
  return e;
}

// 1a. A copied into the LU slot (transposed when stored column-major); identity pivots
template <typename T>
__global__ void __launch_bounds__(BT) k_big_lu_init(const __grid_constant__ UnevenArgs a, const int* __restrict__ list,
                                                    int nlist, int uni_nA, int uni_nT) {
  for (int li = blockIdx.x; li < nlist; li += gridDim.x) {
    const Elem E = elem_of(a, list, li, uni_nA, uni_nT);
    const int nA = E.nA;
    const T* A = reinterpret_cast<const T*>(a.A) + E.o[0];
    T* L = reinterpret_cast<T*>(a.LU) + E.o[0];
    const bool cm = a.colmajor != 0;
    for (size_t i = threadIdx.x; i < (size_t)nA * nA; i += BT) L[i] = cm ? A[(i % nA) * nA + i / nA] : A[i];
    for (int i = threadIdx.x; i < nA; i += BT) a.piv[E.o[3] + i] = i;
  }
}

// 1b. panel jb (columns [j0, j0 + w), rows [j0, nA)) of every element: factorised in shared memory
// (row stride LB + 1), pivots recorded as global rows, the interchanges applied to the other
// columns, and the block row U12 = L11^{-1} A12 right of the panel solved (one thread per column)
template <typename T>
__global__ void __launch_bounds__(BT) k_big_lu_panel(const __grid_constant__ UnevenArgs a, const int* __restrict__ list,
                                                     int nlist, int uni_nA, int uni_nT, int jb) {
  constexpr int LB = lu_panel<T>(), PS = LB + 1;
  extern __shared__ __align__(16) unsigned char lu_smem[];
  T* P = reinterpret_cast<T*>(lu_smem);
  using Key = decltype(abs_key(T(0)));
  __shared__ Key rkey_v[BT / 32];
  __shared__ T s_inv;
  __shared__ int rkey_i[BT / 32];
  __shared__ int spiv[LB];
  __shared__ int s_bad;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  for (int li = blockIdx.x; li < nlist; li += gridDim.x) {
    const Elem E = elem_of(a, list, li, uni_nA, uni_nT);
    const int nA = E.nA, j0 = jb * LB;
    if (j0 >= nA) continue;  // uniform over the CTA
    const int w = min(LB, nA - j0), R = nA - j0;
    T* L = reinterpret_cast<T*>(a.LU) + E.o[0];
    int* piv = a.piv + E.o[3];
    __syncthreads();  // the previous element's panel is free
    for (int i = tid; i < R * w; i += BT) {
      const int r = i / w, c = i % w;
      P[r * PS + c] = L[(size_t)(j0 + r) * nA + j0 + c];
    }
    if (tid == 0) s_bad = 0;
    __syncthreads();
    for (int c = 0; c < w; ++c) {
      Key bv = -1;
      int bi = 0x7fffffff;
      for (int r = c + tid; r < R; r += BT) {
        const Key v = abs_key(P[r * PS + c]);
        if (v > bv || (v == bv && v >= 0 && r < bi)) {
          bv = v;
          bi = r;
        }
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        const Key ov = __shfl_xor_sync(0xffffffffu, bv, off);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
        if (ov > bv || (ov == bv && oi < bi)) {
          bv = ov;
          bi = oi;
        }
      }
      if (lane == 0) {
        rkey_v[wid] = bv;
        rkey_i[wid] = bi;
      }
      __syncthreads();
      if (tid == 0) {
        Key v = rkey_v[0];
        int ii = rkey_i[0];
        for (int q = 1; q < BT / 32; ++q)
          if (rkey_v[q] > v || (rkey_v[q] == v && rkey_i[q] < ii)) {
            v = rkey_v[q];
            ii = rkey_i[q];
          }
        spiv[c] = ii;
        if (!(v > 0))
          s_bad = 1;
        else
          s_inv = T(1) / P[ii * PS + c];  // once: a division by every warp held the FP64 pipe longest
      }
      __syncthreads();
      if (s_bad) break;
      const int pr = spiv[c];
      if (pr != c)
        for (int x = tid; x < w; x += BT) {
          const T u = P[c * PS + x];
          P[c * PS + x] = P[pr * PS + x];
          P[pr * PS + x] = u;
        }
      __syncthreads();
      const T inv = s_inv;
      for (int r = c + 1 + tid; r < R; r += BT) {
        const T l = P[r * PS + c] * inv;
        P[r * PS + c] = l;
        for (int x = c + 1; x < w; ++x) P[r * PS + x] -= l * P[c * PS + x];
      }
      __syncthreads();
    }
    if (s_bad) {
      if (tid == 0) {
        atomicOr(a.status, DEV_ERR_SINGULAR);
        atomicMin(a.status + 1, E.k);
      }
      continue;  // the element's factors are left unfinished; its pivots stay in range
    }
    for (int i = tid; i < R * w; i += BT) {
      const int r = i / w, c = i % w;
      L[(size_t)(j0 + r) * nA + j0 + c] = P[r * PS + c];
    }
    for (int c = tid; c < w; c += BT) piv[j0 + c] = j0 + spiv[c];
    // the interchanges on the columns outside the panel; U12 on those right of it
    for (int col = tid; col < nA - w; col += BT) {
      const int cc = col < j0 ? col : col + w;
      for (int q = 0; q < w; ++q) {
        const int pr = spiv[q];
        if (pr != q) {
          const T u = L[(size_t)(j0 + q) * nA + cc];
          L[(size_t)(j0 + q) * nA + cc] = L[(size_t)(j0 + pr) * nA + cc];
          L[(size_t)(j0 + pr) * nA + cc] = u;
        }
      }
      if (cc >= j0 + w) {
        T x[LB];
#pragma unroll
        for (int q = 0; q < LB; ++q) {
          if (q < w) {
            T v = L[(size_t)(j0 + q) * nA + cc];
#pragma unroll
            for (int s2 = 0; s2 < q; ++s2) v -= P[q * PS + s2] * x[s2];
            x[q] = v;
            L[(size_t)(j0 + q) * nA + cc] = v;
          }
        }
      }
    }
  }
}

// 2-3. X = A^{-1} P [B | r] for a block of CW columns per CTA, whole in shared memory: the permuted
// columns loaded once, forward substitution with the unit lower factor and back substitution with
// the upper factor by panels of SP pivots, X written once.
//
// Bound by the FMA pipe of the block precision (2 nA^2 (nT + 1) flops per element) as far as shared
// memory feeds it.  A panel's update of the other rows runs as tiles of 16 rows x COLG columns per
// warp, each lane holding RPL rows x V columns, so that V 16-byte column vectors and RPL broadcast
// factor vectors from shared memory serve RPL V^2 multiply-adds (128 in FP32; with one row of
// accumulators per lane shared memory took three accesses per multiply-add).  The factor reaches the
// warps through private two-tile rings filled by cp.async one tile ahead, so no block-wide staging
// or barrier stands between tiles; rows and columns beyond nA are zero (unit diagonal), which pads
// every panel to SP pivots.  Rows are interleaved over the lane groups (row G i + g), which with the
// padded ring rows keeps the groups' broadcasts on different banks.  What is left is the in-panel
// solve of a few warps between two barriers and the shared-memory rate of the updates.
// Measured: 4608 FP32 blocks of (320, 480) 40.4 -> 21.7 ms, and 17.8 ms (33 % of the FMA rate) with the
// columns read as vectors, the in-panel rows as four independent chains and the pivots' reciprocals
// formed ahead (of 340 thousand clocks per CTA the load took 55 and the backward in-panel solves 62);
// 750 FP64 blocks
// of (144, 96) 6.28 -> 3.85 ms (74 % of the FP64 rate).  X held in registers instead (one warp per 16
// rows, tile after tile) took 34.8 ms: every tile waits for one warp's chain.
template <typename T, int LC_, int CW_, int NW_, int H_>
struct SolveCfg {
  static constexpr int V = 16 / (int)sizeof(T);      // columns per lane (one 16-byte vector)
  static constexpr int LC = LC_;                     // lanes along the columns
  static constexpr int G = 32 / LC;                  // lane groups along the rows
  static constexpr int RPL = 16 / G;                 // rows per lane
  static constexpr int COLG = LC * V;                // columns of a warp tile
  static constexpr int CW = CW_;                     // columns per CTA
  static constexpr int XST = CW + V;                 // row stride of X
  static constexpr int SP = sizeof(T) == 4 ? 32 : 16;  // pivots per panel
  static constexpr int H = H_;                       // factor tiles per panel
  static constexpr int KT = SP / H;                  // pivots of a factor tile
  static constexpr int UJ = KT * V > 64 ? 2 : KT / V;  // steps of the update unrolled together
  static constexpr int LST = KT + V;                 // its row stride
  static constexpr int NW = NW_;                     // warps per CTA
  static_assert(CW % COLG == 0 && CW <= 32 * NW && SP <= 32, "column groups");
  __host__ __device__ static int rows(int nA) { return (nA + SP - 1) / SP * SP; }
  static size_t smem(int nA) {
    return ((size_t)rows(nA) * XST + (size_t)NW * 2 * 16 * LST + 2 * SP * SP + SP) * sizeof(T) +
           2 * (size_t)rows(nA) * sizeof(int);
  }
};

// dst[r * ld + j] = L[r0 + r][p0 + j], r < nrows, j < W, zero outside the nA x nA factor; vec: rows
// of L start on 16-byte boundaries (nA a multiple of V), copied asynchronously, else by plain loads
template <typename T, int W, int V>
__device__ __forceinline__ void solve_tile(T* dst, int ld, const T* L, int nA, int r0, int p0, int nrows, bool vec,
                                           int t, int nt) {
  if (vec) {
    for (int i = t; i < nrows * (W / V); i += nt) {
      const int r = i / (W / V), q = (i % (W / V)) * V;
      const bool in = r0 + r < nA && p0 + q < nA;
      const T* src = L + (in ? (size_t)(r0 + r) * nA + p0 + q : 0);
      const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst + r * ld + q);
      const int bytes = in ? 16 : 0;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
    }
  } else {
    for (int i = t; i < nrows * W; i += nt) {
      const int r = i / W, j = i % W;
      dst[r * ld + j] = (r0 + r < nA && p0 + j < nA) ? L[(size_t)(r0 + r) * nA + p0 + j] : T(0);
    }
  }
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
template <typename T>
struct alignas(16) SolveVec {
  T v[16 / sizeof(T)];
};

// x / d with inv = 1 / d (rounded) known: the product, then one correction by its remainder, the
// quotient step of P. W. Markstein, "Computation of elementary functions on the IBM RISC System/6000
// processor", IBM J. Res. Dev. 34 (1990).  It takes the division's instruction sequence off the
// substitution's serial chain.  With unit roundoff u the product is within 2 u of x / d (at most two
// units in the last place, not the one that would make the corrected quotient correctly rounded
// always); the remainder leaves the fused multiply-add with a relative error of u and the correction
// adds another, so that the result is within half a unit plus a few u of one.  Outside the
// following the caller divides:
//   * the result is not finite (the reciprocal or a product left the range);
//   * 0 < |x| < 2^8 times the smallest normal number, where the remainder would lose bits to underflow
//     (2^-8 of a unit at the bound, whole units below).
template <typename T>
__device__ __forceinline__ T solve_div(T x, T d, T inv) {
  const T q = x * inv;
  return fma(fma(-q, d, x), inv, q);
}
// that range of x as one integer comparison of a minimum over the values: key(x) < SOLVE_TINY (zero has
// the largest key)
__device__ __forceinline__ unsigned solve_key(float x) { return 2u * __float_as_uint(x) - 1u; }
__device__ __forceinline__ unsigned solve_key(double x) {
  return (2u * (unsigned)__double2hiint(x) | (__double2loint(x) != 0 ? 1u : 0u)) - 1u;
}
template <typename T>
constexpr unsigned SOLVE_TINY = sizeof(T) == 4 ? (9u << 24) - 1u : (9u << 21) - 1u;

template <typename T, int LC, int CW, int NW, int H>
__global__ void __launch_bounds__(32 * NW, 512 / (32 * NW)) k_big_solve(const __grid_constant__ UnevenArgs a, const int* __restrict__ list,
                                                  int base, int nlist, int uni_nA, int uni_nT) {
  using C = SolveCfg<T, LC, CW, NW, H>;
  constexpr int V = C::V, G = C::G, RPL = C::RPL, COLG = C::COLG, XST = C::XST, SP = C::SP, KT = C::KT, LST = C::LST;
  constexpr int NTH = 32 * NW;
  extern __shared__ __align__(16) unsigned char sv_smem[];
  if ((int)blockIdx.y >= nlist) return;
  const Elem E = elem_of(a, list, base + blockIdx.y, uni_nA, uni_nT);
  const int nA = E.nA, nT = E.nT, c0 = blockIdx.x * CW;
  if (c0 > nT) return;  // uniform over the CTA (column nT is r: x_r)
  const int nAp = C::rows(nA);
  T* Xs = reinterpret_cast<T*>(sv_smem);            // nAp x XST
  T* ring = Xs + (size_t)nAp * XST;                  // NW x 2 factor tiles of 16 x LST
  T* Dg = ring + (size_t)NW * 2 * 16 * LST;          // two diagonal blocks SP x SP
  T* dinv = Dg + 2 * SP * SP;                        // reciprocals of a panel's pivots
  int* perm = reinterpret_cast<int*>(dinv + SP);
  int* pvs = perm + nAp;
  const T* L = reinterpret_cast<const T*>(a.LU) + E.o[0];
  const T* B = reinterpret_cast<const T*>(a.B) + E.o[1];
  T* X = reinterpret_cast<T*>(a.XB) + E.o[1];
  const int* piv = a.piv + E.o[3];
  const bool cm = a.colmajor != 0;
  const bool vec = nA % V == 0 && (reinterpret_cast<uintptr_t>(L) & 15) == 0;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int live = min(CW, nT + 1 - c0);             // columns of this CTA, r included
  const int ncg = (live + COLG - 1) / COLG;
  T* tile = ring + (size_t)wid * 2 * 16 * LST;
  const int np = nAp / SP;
  // the factor tile of this warp's first unit of a panel and the first diagonal block
  auto first_tile = [&](int ra, int rows, int p0) {
    if (wid < rows / 16 * ncg) solve_tile<T, KT, V>(tile, LST, L, nA, ra + 16 * (wid / ncg), p0, 16, vec, lane, 32);
    cp_commit();
  };
  solve_tile<T, SP, V>(Dg, SP, L, nA, 0, 0, SP, vec, tid, NTH);
  cp_commit();
  // position i of P b holds row perm[i]: the interchanges (j, piv[j]) undone from the last to the
  // first, every position on its own.  Where columns are read along the rows (column-major B), perm
  // is the position of a row instead.
  const bool vecb = (cm ? nA : nT) % V == 0 && (reinterpret_cast<uintptr_t>(B) & 15) == 0;
  const bool inverse = cm && vecb;
  for (int i = tid; i < nAp; i += NTH) {
    const int p = i < nA ? piv[i] : i;
    pvs[i] = p >= 0 && p < nA ? p : i;
  }
  __syncthreads();
  for (int i = tid; i < nAp; i += NTH) {
    int pos = i;
    for (int j = nAp - 4; j >= 0; j -= 4) {
      const int4 p = *reinterpret_cast<const int4*>(pvs + j);
      pos = pos == j + 3 ? p.w : (pos == p.w ? j + 3 : pos);
      pos = pos == j + 2 ? p.z : (pos == p.z ? j + 2 : pos);
      pos = pos == j + 1 ? p.y : (pos == p.y ? j + 1 : pos);
      pos = pos == j ? p.x : (pos == p.x ? j : pos);
    }
    perm[inverse ? pos : i] = inverse ? i : pos;
  }
  __syncthreads();
  // the permuted columns.  Column-major B: a warp reads two vectors of rows of 16 columns (whole
  // sectors), SU such reads in flight, and stores each value at its row's position (conflict-free
  // without interchanges); row-major: rows by 16-byte asynchronous copies; one value per lane where
  // rows or columns do not start on vectors
  constexpr int SU = 8;
  const double* rv = a.r + E.o[3];
  if (inverse) {
    const int nr = nAp / (2 * V), ni = nr * (CW / 16);
    for (int i0 = wid; i0 < ni; i0 += NW * SU) {
      SolveVec<T> v[SU];
#pragma unroll
      for (int u = 0; u < SU; ++u) {
        const int it = i0 + NW * u, iq = it / nr, row = (2 * (it - iq * nr) + (lane >> 4)) * V;
        const int c = c0 + iq * 16 + (lane & 15);
#pragma unroll
        for (int e = 0; e < V; ++e) v[u].v[e] = T(0);
        if (it < ni && row < nA) {
          if (c < nT) {
            v[u] = *reinterpret_cast<const SolveVec<T>*>(B + (size_t)c * nA + row);
          } else if (c == nT) {
#pragma unroll
            for (int e = 0; e < V; ++e) v[u].v[e] = T(rv[row + e]);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < SU; ++u) {
        const int it = i0 + NW * u, iq = it / nr, row = (2 * (it - iq * nr) + (lane >> 4)) * V;
        if (it < ni)
#pragma unroll
          for (int e = 0; e < V; ++e) Xs[(size_t)perm[row + e] * XST + iq * 16 + (lane & 15)] = v[u].v[e];
      }
    }
  } else if (vecb) {
    constexpr int LV = CW / V, RW = 32 / LV;  // lanes per row, rows per warp
    const int q = lane % LV * V, c = c0 + q;
    for (int i = wid * RW + lane / LV; i < nAp; i += NW * RW) {
      T* dst = Xs + (size_t)i * XST + q;
      if (i < nA && c < nT) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                     "l"(B + (size_t)perm[i] * nT + c)
                     : "memory");
      } else {
        SolveVec<T> z;
#pragma unroll
        for (int e = 0; e < V; ++e) z.v[e] = T(0);
        if (i < nA && c == nT) z.v[0] = T(rv[perm[i]]);
        *reinterpret_cast<SolveVec<T>*>(dst) = z;
      }
    }
    cp_commit();
  } else {
    const int nr = cm ? nAp / 8 : nAp, ni = cm ? nr * (CW / 4) : nr * (CW / 32 + (CW % 32 != 0));
    for (int it = wid; it < ni; it += NW) {
      const int ir = it % nr, iq = it / nr;
      const int i = cm ? ir * 8 + (lane & 7) : ir, q = cm ? iq * 4 + (lane >> 3) : iq * 32 + lane;
      const int c = c0 + q;
      if (q >= CW) continue;
      T v = T(0);
      if (i < nA) {
        const int src = perm[i];
        v = c < nT ? B[cm ? (size_t)c * nA + src : (size_t)src * nT + c] : (c == nT ? T(rv[src]) : T(0));
      }
      Xs[(size_t)i * XST + q] = v;
    }
  }
  // rows [ra, ra + rows) of X -= (factor rows, columns p0 ..) x (solved rows p0 ..); the first tile is
  // on its way
  auto update = [&](int ra, int rows, int p0) {
    const int units = rows / 16 * ncg;
    const int g = lane / LC, lc = lane % LC;
    int slot = 0;
    for (int u = wid; u < units; u += NW) {
      T* xo = Xs + (size_t)(ra + 16 * (u / ncg) + g) * XST + (u % ncg) * COLG + lc * V;
      T acc[RPL][V];
#pragma unroll
      for (int i = 0; i < RPL; ++i)
#pragma unroll
        for (int q = 0; q < V; ++q) acc[i][q] = T(0);
#pragma unroll
      for (int h = 0; h < H; ++h, slot ^= 1) {  // tile h of the panel's pivots; the next one on its way
        const int un = h + 1 < H ? u : u + NW;
        if (un < units)
          solve_tile<T, KT, V>(tile + (slot ^ 1) * 16 * LST, LST, L, nA, ra + 16 * (un / ncg), p0 + (h + 1) % H * KT,
                               16, vec, lane, 32);
        cp_commit();
        cp_wait<1>();
        __syncwarp();
        const T* lt = tile + slot * 16 * LST + g * LST;
        const T* xp = Xs + (size_t)(p0 + h * KT) * XST + (u % ncg) * COLG + lc * V;
#pragma unroll(C::UJ)
        for (int j = 0; j < KT; j += V) {
          SolveVec<T> xv[V];
#pragma unroll
          for (int s = 0; s < V; ++s) xv[s] = *reinterpret_cast<const SolveVec<T>*>(xp + (size_t)(j + s) * XST);
#pragma unroll
          for (int i = 0; i < RPL; ++i) {
            const SolveVec<T> l = *reinterpret_cast<const SolveVec<T>*>(lt + G * i * LST + j);
#pragma unroll
            for (int s = 0; s < V; ++s)
#pragma unroll
              for (int q = 0; q < V; ++q) acc[i][q] = fma(l.v[s], xv[s].v[q], acc[i][q]);
          }
        }
        __syncwarp();  // the slot may be refilled
      }
#pragma unroll
      for (int i = 0; i < RPL; ++i) {
        SolveVec<T>* xr = reinterpret_cast<SolveVec<T>*>(xo + (size_t)G * i * XST);
        SolveVec<T> x = *xr;
#pragma unroll
        for (int q = 0; q < V; ++q) x.v[q] -= acc[i][q];
        *xr = x;
      }
    }
    cp_wait<0>();
  };
  // ---- forward: unit lower factor, panels top to bottom
  for (int pb = 0; pb < np; ++pb) {
    const int p0 = pb * SP, ra = p0 + SP, rows = nAp - ra;
    const T* D = Dg + (pb & 1) * SP * SP;
    first_tile(ra, rows, p0);
    cp_wait<1>();     // the diagonal block
    __syncthreads();  // and the rows of the panel are final
    if (tid < live) {  // in-panel solve, one column per thread, the panel's rows in registers
      T x[SP];
#pragma unroll
      for (int r = 0; r < SP; ++r) x[r] = Xs[(size_t)(p0 + r) * XST + tid];
      // four rows at a time: their sums over the solved rows are independent chains
#pragma unroll
      for (int rb = 0; rb < SP; rb += 4) {
#pragma unroll
        for (int c = 0; c < rb; c += V) {
          SolveVec<T> l[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) l[i] = *reinterpret_cast<const SolveVec<T>*>(D + (rb + i) * SP + c);
#pragma unroll
          for (int s = 0; s < V; ++s)
#pragma unroll
            for (int i = 0; i < 4; ++i) x[rb + i] = fma(-l[i].v[s], x[c + s], x[rb + i]);
        }
#pragma unroll
        for (int i = 1; i < 4; ++i)
#pragma unroll
          for (int c = 0; c < i; ++c) x[rb + i] = fma(-D[(rb + i) * SP + rb + c], x[rb + c], x[rb + i]);
      }
#pragma unroll
      for (int r = 0; r < SP; ++r) Xs[(size_t)(p0 + r) * XST + tid] = x[r];
    }
    __syncthreads();
    if (pb + 1 < np)  // the next panel's diagonal block
      solve_tile<T, SP, V>(Dg + ((pb + 1) & 1) * SP * SP, SP, L, nA, ra, ra, SP, vec, tid, NTH);
    cp_commit();
    update(ra, rows, p0);
  }
  // ---- backward: upper factor, panels bottom to top (the last diagonal block is still in place)
  for (int pb = np - 1; pb >= 0; --pb) {
    const int p0 = pb * SP;
    const T* D = Dg + (pb & 1) * SP * SP;
    first_tile(0, p0, p0);
    cp_wait<1>();
    __syncthreads();
    if (32 * wid < live) {  // whole warps
      const int q = min(tid, CW - 1);
      if (lane < SP) dinv[lane] = T(1) / (p0 + lane < nA ? D[lane * SP + lane] : T(1));
      T x[SP];
#pragma unroll
      for (int r = 0; r < SP; ++r) x[r] = Xs[(size_t)(p0 + r) * XST + q];
      __syncwarp();
      bool fin = true;
      unsigned least = ~0u;
#pragma unroll
      for (int rb = SP - 4; rb >= 0; rb -= 4) {
#pragma unroll
        for (int c = SP - V; c >= rb + 4; c -= V) {
          SolveVec<T> l[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) l[i] = *reinterpret_cast<const SolveVec<T>*>(D + (rb + i) * SP + c);
#pragma unroll
          for (int s = V - 1; s >= 0; --s)
#pragma unroll
            for (int i = 3; i >= 0; --i) x[rb + i] = fma(-l[i].v[s], x[c + s], x[rb + i]);
        }
#pragma unroll
        for (int i = 3; i >= 0; --i) {
#pragma unroll
          for (int c = 3; c > i; --c) x[rb + i] = fma(-D[(rb + i) * SP + rb + c], x[rb + c], x[rb + i]);
          least = min(least, solve_key(x[rb + i]));
          x[rb + i] = solve_div<T>(x[rb + i], D[(rb + i) * SP + rb + i], dinv[rb + i]);
          fin = fin && isfinite(x[rb + i]);
        }
      }
      if (__any_sync(0xffffffffu, !fin || least < SOLVE_TINY<T>)) {  // out of range somewhere: the columns again, by divisions
        if (tid < CW)
          for (int r = SP - 1; r >= 0; --r) {
            T* xr = Xs + (size_t)(p0 + r) * XST + tid;
            T v = *xr;
            for (int c = SP - 1; c > r; --c) v = fma(-D[r * SP + c], xr[(size_t)(c - r) * XST], v);
            *xr = p0 + r < nA ? v / D[r * SP + r] : v;
          }
      } else if (tid < CW) {
#pragma unroll
        for (int r = 0; r < SP; ++r) Xs[(size_t)(p0 + r) * XST + tid] = x[r];
      }
    }
    __syncthreads();
    if (pb > 0)
      solve_tile<T, SP, V>(Dg + ((pb - 1) & 1) * SP * SP, SP, L, nA, p0 - SP, p0 - SP, SP, vec, tid, NTH);
    cp_commit();
    update(0, p0, p0);
  }
  __syncthreads();
  for (int it = tid; it < nA * CW; it += NTH) {
    const int i = it / CW, q = it % CW, c = c0 + q;
    if (c < nT)
      X[(size_t)i * nT + c] = Xs[(size_t)i * XST + q];
    else if (c == nT)
      a.xr[E.o[3] + i] = double(Xs[(size_t)i * XST + q]);
  }
}

// 1c / 4. batched GEMM Out -= A B, per element:
//   phase 2: S = D - C X_B (C, D column-major when the blocks are)
//   phase 3: L[j1:, j1:] -= L[j1:, j0:j1] L[j0:j1, j1:]          (LU trailing update, panel jb)
// 16 x 16 threads, each with TM x TM outputs in two TM/2-wide halves of rows and of columns (so
// that its shared-memory operands are two 16-byte vectors per k), GKK values of k per stage, two
// shared-memory stages with the next stage's global values held in registers meanwhile.
template <typename T>
struct GemmCfg {
  // outputs per thread and dimension.  FP64: 32 x 32 tiles, so that blocks of 96 to 144 leave few idle
  // lanes (64 x 64 tiles computed 16 384 outputs for the 9 216 of a 96 x 96 block); the FP64 pipe, not
  // the shared memory that a larger tile saves, is the limit
  static constexpr int TM = sizeof(T) == 8 ? 2 : 8;
  static constexpr int H = TM / 2;                   // FP32: one 16-byte vector
  static constexpr int BM = 16 * TM;                 // output tile (rows = columns)
  static constexpr int GKK = 8;                      // k per stage
  static constexpr int PAD = 16 / sizeof(T);
  static constexpr int LD = BM * GKK / BT;           // values of each operand a thread loads per stage
};
template <typename T>
__device__ __forceinline__ void gemm_vec_ld(const T* p, T (&v)[GemmCfg<T>::H]) {
  if constexpr (sizeof(T) == 8) {
    v[0] = *p;
  } else {
    const float4 x = *reinterpret_cast<const float4*>(p);
    v[0] = x.x;
    v[1] = x.y;
    v[2] = x.z;
    v[3] = x.w;
  }
}
template <typename T>
__global__ void __launch_bounds__(BT) k_big_gemm(const __grid_constant__ UnevenArgs a, const int* __restrict__ list,
                                                 int base, int nlist, int uni_nA, int uni_nT, int phase, int jb) {
  using C = GemmCfg<T>;
  constexpr int TM = C::TM, H = C::H, BM = C::BM, GKK = C::GKK, LDN = C::LD;
  __shared__ __align__(16) T As[2][GKK][BM + C::PAD];  // [k][m]
  __shared__ __align__(16) T Bs[2][GKK][BM + C::PAD];  // [k][n]
  if ((int)blockIdx.z >= nlist) return;
  const int li = base + blockIdx.z;
  const Elem E = elem_of(a, list, li, uni_nA, uni_nT);
  const int nA = E.nA, nT = E.nT;
  const bool cm = a.colmajor != 0;
  int M, N, K, m_off = 0, k_off = 0, n_off = 0;
  T* L = reinterpret_cast<T*>(a.LU) + E.o[0];
  T* X = reinterpret_cast<T*>(a.XB) + E.o[1];
  const T* Cm = reinterpret_cast<const T*>(a.C) + E.o[1];
  const T* Dm = reinterpret_cast<const T*>(a.D) + E.o[2];
  T* S = reinterpret_cast<T*>(a.S) + E.o[2];
  if (phase == 2) {
    M = nT;
    N = nT;
    K = nA;
  } else {
    const int j0 = jb * lu_panel<T>(), j1 = min(nA, j0 + lu_panel<T>());
    M = nA - j1;
    N = nA - j1;
    K = j1 - j0;
    m_off = j1;
    n_off = j1;
    k_off = j0;
  }
  const int tm0 = blockIdx.y * BM, tn0 = blockIdx.x * BM;
  if (M <= 0 || K <= 0 || tm0 >= M || tn0 >= N) return;
  const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
  // operand A element (m, k) of the tile: k contiguous in memory except column-major C
  const bool a_mfast = phase == 2 && cm;
  auto lda = [&](int m, int k) -> T {
    if (m >= M || k >= K) return T(0);
    if (phase != 2) return L[(size_t)(m_off + m) * nA + k_off + k];
    return cm ? Cm[(size_t)k * nT + m] : Cm[(size_t)m * nA + k];
  };
  auto ldb = [&](int k, int n) -> T {
    if (n >= N || k >= K) return T(0);
    return phase == 3 ? L[(size_t)(k_off + k) * nA + n_off + n] : X[(size_t)(k_off + k) * nT + n];
  };
  // thread's load slots: A (m, k) with k fastest (or m fastest), B (k, n) with n fastest
  T ra[LDN], rb[LDN];
  auto gload = [&](int k0) {
#pragma unroll
    for (int q = 0; q < LDN; ++q) {
      const int idx = tid + q * BT;
      if (a_mfast)
        ra[q] = lda(tm0 + idx % BM, k0 + idx / BM);
      else
        ra[q] = lda(tm0 + idx / GKK, k0 + idx % GKK);
      rb[q] = ldb(k0 + idx / BM, tn0 + idx % BM);
    }
  };
  auto sstore = [&](int st) {
#pragma unroll
    for (int q = 0; q < LDN; ++q) {
      const int idx = tid + q * BT;
      if (a_mfast)
        As[st][idx / BM][idx % BM] = ra[q];
      else
        As[st][idx % GKK][idx / GKK] = ra[q];
      Bs[st][idx / BM][idx % BM] = rb[q];
    }
  };
  T acc[TM][TM];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TM; ++j) acc[i][j] = T(0);
  gload(0);
  sstore(0);
  __syncthreads();
  int st = 0;
  for (int k0 = 0; k0 < K; k0 += GKK) {
    const bool more = k0 + GKK < K;
    if (more) gload(k0 + GKK);
#pragma unroll
    for (int kk = 0; kk < GKK; ++kk) {
      T av[TM], bv[TM];
      gemm_vec_ld<T>(&As[st][kk][ty * H], *reinterpret_cast<T(*)[H]>(&av[0]));
      gemm_vec_ld<T>(&As[st][kk][BM / 2 + ty * H], *reinterpret_cast<T(*)[H]>(&av[H]));
      gemm_vec_ld<T>(&Bs[st][kk][tx * H], *reinterpret_cast<T(*)[H]>(&bv[0]));
      gemm_vec_ld<T>(&Bs[st][kk][BM / 2 + tx * H], *reinterpret_cast<T(*)[H]>(&bv[H]));
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TM; ++j) acc[i][j] += av[i] * bv[j];
    }
    if (more) {
      sstore(st ^ 1);
      __syncthreads();
      st ^= 1;
    }
  }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int m = tm0 + (i < H ? ty * H + i : BM / 2 + ty * H + i - H);
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < TM; ++j) {
      const int n = tn0 + (j < H ? tx * H + j : BM / 2 + tx * H + j - H);
      if (n >= N) continue;
      if (phase == 3) {
        L[(size_t)(m_off + m) * nA + n_off + n] -= acc[i][j];
      } else {
        const T d = cm ? Dm[(size_t)n * nT + m] : Dm[(size_t)m * nT + n];
        S[(size_t)m * nT + n] = d - acc[i][j];
      }
    }
  }
}

// 4'. S = D - C X_B of FP32 blocks on the tensor cores (tcgen05, 3xTF32: each operand split into a
// TF32 high part and the remainder, hi*hi + hi*lo + lo*hi accumulated in FP32 in tensor memory).
// One CTA per output tile of TM rows (m) x 128 columns (n) of one element, computed transposed: the
// tensor-memory lanes hold the 128 columns n and its TM FP32 columns the rows m, so that in the
// epilogue the 32 lanes of a warp write 32 consecutive n of one row (coalesced).  K runs in chunks
// of KC staged K-major without swizzle (hfr_tc.cuh) in two shared-memory buffers, one mbarrier per
// buffer; the next chunk's global loads are in flight while the tensor core works on the current
// one.  A thread stages four consecutive k of a row as one 16-byte store, and the eight threads of a
// store's quarter-warp write the eight rows of one core matrix: 128 contiguous bytes, free of bank
// conflicts (single-value stores of the same layout met four to a bank and set the kernel's time).
// Measured: 4608 blocks of (320, 480) 14.7 -> 6.1 ms, the p = 4 and 5 blocks of a wall mesh (10 000
// elements) 1.71 -> 0.20 ms.  KC = 16 leaves two CTAs per SM (TM = 256) or three (TM = 128, taken when nT <= 128), so that one
// CTA's epilogue runs under another's products.
namespace btc {
constexpr int TN = 128, KC = 16, THREADS = 256;
constexpr uint32_t SBO = (KC / 4) * 128u;
constexpr uint32_t N_BYTES = (TN / 8) * SBO;  // the n-rows operand (MMA A, 128 rows), hi or lo
template <int TM>
__host__ __device__ constexpr uint32_t m_bytes() { return (TM / 8) * SBO; }  // the m-rows operand (MMA B), hi or lo
template <int TM>
__host__ __device__ constexpr uint32_t stage() { return 2 * N_BYTES + 2 * m_bytes<TM>(); }
template <int TM>
__host__ __device__ constexpr uint32_t smem() { return 2 * stage<TM>() + 64; }
static_assert(smem<256>() <= 232448 / 2, "two CTAs per SM");
__device__ __forceinline__ void split_store(unsigned char* hi, unsigned char* lo, uint32_t o, const float (&v)[4]) {
  float h[4], l[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) tc::split_tf32(v[e], h[e], l[e]);
  *reinterpret_cast<float4*>(hi + o) = make_float4(h[0], h[1], h[2], h[3]);
  *reinterpret_cast<float4*>(lo + o) = make_float4(l[0], l[1], l[2], l[3]);
}
}  // namespace btc

template <int TM>
__global__ void __launch_bounds__(btc::THREADS, 2) k_big_s_tc(const __grid_constant__ UnevenArgs a,
                                                             const int* __restrict__ list, int base, int nlist,
                                                             int uni_nA, int uni_nT) {
  using namespace tc;
  using namespace btc;
  extern __shared__ __align__(1024) unsigned char btc_smem[];
  if ((int)blockIdx.z >= nlist) return;
  const Elem E = elem_of(a, list, base + blockIdx.z, uni_nA, uni_nT);
  const int nT = E.nT, K = E.nA;
  const bool cm = a.colmajor != 0;
  const float* X = reinterpret_cast<const float*>(a.XB) + E.o[1];
  const float* Cm = reinterpret_cast<const float*>(a.C) + E.o[1];
  const float* Dm = reinterpret_cast<const float*>(a.D) + E.o[2];
  float* S = reinterpret_cast<float*>(a.S) + E.o[2];
  const int tm0 = blockIdx.y * TM, tn0 = blockIdx.x * TN;
  if (tm0 >= nT || tn0 >= nT) return;  // uniform over the CTA
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  constexpr uint32_t MB = m_bytes<TM>(), STAGE = stage<TM>();
  uint64_t* mbar = reinterpret_cast<uint64_t*>(btc_smem + 2 * STAGE);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(mbar + 2);
  if (t == 0) {
    mbar_init(smem_u32(mbar), 1);
    mbar_init(smem_u32(mbar + 1), 1);
  }
  if (w == 0) tmem_alloc(smem_u32(tslot), TM);
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = *tslot;
  const int NM = min(TM, (nT - tm0 + 15) & ~15);  // rows m that the products cover
  const bool avec = !cm && K % 4 == 0 && (reinterpret_cast<uintptr_t>(Cm) & 15) == 0;
  // staging: column n = t & 127 of X, k quads (t >> 7) + 2 u; rows of C: column-major one row per
  // thread (row t % TM, quads t / TM + (256 / TM) u), row-major eight rows x four quads per warp
  constexpr int QN = KC / 8;           // quads of X per thread
  constexpr int QM = TM * KC / 1024;   // quads of C per thread
  float rb[QN][4], ra[QM][4];
  auto gload = [&](int k0) {
#pragma unroll
    for (int u = 0; u < QN; ++u) {
      const int n = tn0 + (t & 127), k = k0 + 4 * ((t >> 7) + 2 * u);
#pragma unroll
      for (int e = 0; e < 4; ++e) rb[u][e] = (n < nT && k + e < K) ? X[(size_t)(k + e) * nT + n] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < QM; ++u) {
      if (cm) {
        const int m = tm0 + t % TM, k = k0 + 4 * (t / TM + (THREADS / TM) * u);
#pragma unroll
        for (int e = 0; e < 4; ++e) ra[u][e] = (m < nT && k + e < K) ? Cm[(size_t)(k + e) * nT + m] : 0.f;
      } else {
        const int m = tm0 + 64 * u + 8 * w + (lane & 7), k = k0 + 4 * (lane >> 3);
        if (avec) {
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
          if (m < nT && k < K) v = *reinterpret_cast<const float4*>(Cm + (size_t)m * K + k);
          ra[u][0] = v.x;
          ra[u][1] = v.y;
          ra[u][2] = v.z;
          ra[u][3] = v.w;
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) ra[u][e] = (m < nT && k + e < K) ? Cm[(size_t)m * K + k + e] : 0.f;
        }
      }
    }
  };
  auto sstore = [&](int b) {
    unsigned char* Nhi = btc_smem + b * STAGE;
    unsigned char* Mhi = Nhi + 2 * N_BYTES;
#pragma unroll
    for (int u = 0; u < QN; ++u)
      split_store(Nhi, Nhi + N_BYTES, kmajor_offset(t & 127, 4 * ((t >> 7) + 2 * u), SBO), rb[u]);
#pragma unroll
    for (int u = 0; u < QM; ++u) {
      const int m = cm ? t % TM : 64 * u + 8 * w + (lane & 7);
      const int k = cm ? 4 * (t / TM + (THREADS / TM) * u) : 4 * (lane >> 3);
      split_store(Mhi, Mhi + MB, kmajor_offset(m, k, SBO), ra[u]);
    }
  };
  const int nch = (K + KC - 1) / KC;
  const uint32_t idesc = idesc_tf32(TN, NM);  // M = 128 (n on the lanes), N = NM (m)
  bool ok = true;
  gload(0);
  for (int c = 0; c < nch; ++c) {
    const int b = c & 1;
    if (c >= 2) {  // the MMAs of chunk c - 2 read this buffer
      ok = mbar_wait(smem_u32(mbar + b), (uint32_t)(((c - 2) >> 1) & 1), TIMEOUT_NS);
      if (__syncthreads_or(!ok)) {
        ok = false;
        break;
      }
      fence_after_sync();
    }
    sstore(b);
    fence_proxy_async();
    fence_before_sync();
    __syncthreads();
    if (t == 0) {
      fence_after_sync();
      const uint32_t nh = smem_u32(btc_smem + b * STAGE), nl = nh + N_BYTES, mh = nl + N_BYTES, ml = mh + MB;
#pragma unroll 1
      for (int kk = 0; kk < KC / 8; ++kk) {
        const uint32_t off = (uint32_t)kk * 256u;  // two core matrices along k per instruction
        const uint32_t acc = (c > 0 || kk > 0) ? 1u : 0u;
        mma_tf32(tmem, desc_noswizzle(nh + off, 128, SBO), desc_noswizzle(mh + off, 128, SBO), idesc, acc);
        mma_tf32(tmem, desc_noswizzle(nh + off, 128, SBO), desc_noswizzle(ml + off, 128, SBO), idesc, 1u);
        mma_tf32(tmem, desc_noswizzle(nl + off, 128, SBO), desc_noswizzle(mh + off, 128, SBO), idesc, 1u);
      }
      mma_commit(smem_u32(mbar + b));
    }
    if (c + 1 < nch) gload((c + 1) * KC);
  }
  if (ok) {  // the last commit completes after every MMA before it
    ok = mbar_wait(smem_u32(mbar + ((nch - 1) & 1)), (uint32_t)(((nch - 1) >> 1) & 1), TIMEOUT_NS);
    ok = !__syncthreads_or(!ok);
  }
  fence_after_sync();
  if (ok) {
    // warp w: lanes 32 (w % 4) .., every other group of 16 rows; a column-major D is contiguous along
    // a thread's rows (16-byte loads), a row-major one along the lanes
    const int q = w & 3;
    const int n = tn0 + 32 * q + lane;
    const uint32_t tl = (uint32_t)(32 * q) << 16;
    const bool dvec = cm && nT % 4 == 0 && (reinterpret_cast<uintptr_t>(Dm) & 15) == 0;
#pragma unroll 1
    for (int cc = w >> 2; cc < NM / 16; cc += 2) {
      float v[16], d[16];
      const int m0 = tm0 + 16 * cc;
#pragma unroll
      for (int u = 0; u < 16; u += 4) {
        if (dvec) {
          float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
          if (n < nT && m0 + u < nT) x = *reinterpret_cast<const float4*>(Dm + (size_t)n * nT + m0 + u);
          d[u] = x.x;
          d[u + 1] = x.y;
          d[u + 2] = x.z;
          d[u + 3] = x.w;
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int m = m0 + u + e;
            d[u + e] = (n < nT && m < nT) ? (cm ? Dm[(size_t)n * nT + m] : Dm[(size_t)m * nT + n]) : 0.f;
          }
        }
      }
      tmem_ld16(tmem + tl + (uint32_t)(16 * cc), v);
      if (n >= nT) continue;
#pragma unroll
      for (int u = 0; u < 16; ++u)
        if (m0 + u < nT) S[(size_t)(m0 + u) * nT + n] = d[u] - v[u];
    }
  } else if (t == 0) {
    atomicOr(a.status, DEV_ERR_TIMEOUT);
    // the MMAs in flight finish (bounded) before their tensor memory is released
    mbar_wait(smem_u32(mbar), 0, TIMEOUT_NS);
    mbar_wait(smem_u32(mbar + 1), 0, TIMEOUT_NS);
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  if (w == 0) tmem_dealloc(tmem, TM);
}

// rows of FP32 blocks up to which x_r comes in FP32 with X: the accumulated rounding of a substitution
// grows with the rows, and above this r stays in FP64 throughout (24 blocks of 1024 rows: error of x_r
// 4.2e-7 of the largest value, rms 3.8e-8; 894 rows, in FP32: 5.7e-7, rms 6.5e-8)
constexpr int XR32_MAX = 894;

// y = U^{-1} L^{-1} P r in FP64 with the stored factors (row-major, unit lower L), y and pvs in shared
// memory, one CTA: by panels of 32 rows, the products with the solved rows a row per warp (lanes along
// it), then the panel's own triangle by one warp, a row per lane
template <typename T>
__device__ void xr_solve(const T* L, const int* piv, const double* r, int nA, double* y, int* pvs) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < nA; i += BT) {
    const int p = piv[i];
    pvs[i] = p >= 0 && p < nA ? p : i;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nA; i += BT) {  // position i of P r: the interchanges from the last to the first
    int pos = i;
    for (int j = nA - 1; j >= 0; --j) {
      const int p = pvs[j];
      pos = pos == j ? p : (pos == p ? j : pos);
    }
    y[i] = r[pos];
  }
  __syncthreads();
  const int np = (nA + 31) / 32;
  for (int dir = 0; dir < 2; ++dir) {
    for (int q = 0; q < np; ++q) {
      const int p0 = 32 * (dir == 0 ? q : np - 1 - q), c0 = dir == 0 ? 0 : p0 + 32, c1 = dir == 0 ? p0 : nA;
      for (int row = p0 + wid; row < min(p0 + 32, nA); row += BT / 32) {
        double s = 0.0;
        for (int c = c0 + lane; c < c1; c += 32) s = fma((double)L[(size_t)row * nA + c], y[c], s);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) y[row] -= s;
      }
      __syncthreads();
      if (wid == 0) {
        const int row = p0 + lane, n = min(32, nA - p0);
        const T* Lr = L + (size_t)(row < nA ? row : p0) * nA + p0;
        double v = row < nA ? y[row] : 0.0;
        for (int k = 0; k < n; ++k) {
          const int c = dir == 0 ? k : n - 1 - k;
          if (dir == 1 && lane == c) v /= (double)Lr[c];
          const double yc = __shfl_sync(0xffffffffu, v, c);
          if (row < nA && (dir == 0 ? lane > c : lane < c)) v -= (double)Lr[c] * yc;
        }
        if (row < nA) y[row] = v;
      }
      __syncthreads();
    }
  }
}

// 5. t = s - C x_r.  XR: x_r by the FP64 substitution above, else as it came with X (the right-hand
// side's column of the column-block solve)
template <typename T, bool XR>
__global__ void __launch_bounds__(BT) k_big_t(const __grid_constant__ UnevenArgs a, const int* __restrict__ list,
                                              int nlist, int uni_nA, int uni_nT) {
  __shared__ double y[1024];
  __shared__ int pvs[XR ? 1024 : 1];
  for (int li = blockIdx.x; li < nlist; li += gridDim.x) {
    const Elem E = elem_of(a, list, li, uni_nA, uni_nT);
    const int nA = E.nA, nT = E.nT;
    const T* Cm = reinterpret_cast<const T*>(a.C) + E.o[1];
    double* xr = a.xr + E.o[3];
    const double* sv = a.s + E.o[4];
    double* t = a.t + E.o[4];
    const bool cm = a.colmajor != 0;
    __syncthreads();
    if constexpr (XR) {
      xr_solve<T>(reinterpret_cast<const T*>(a.LU) + E.o[0], a.piv + E.o[3], a.r + E.o[3], nA, y, pvs);
      for (int i = threadIdx.x; i < nA; i += BT) xr[i] = y[i];
    } else {
      for (int i = threadIdx.x; i < nA; i += BT) y[i] = xr[i];
      __syncthreads();
    }
    for (int row = threadIdx.x; row < nT; row += BT) {
      double acc = 0.0;
      for (int c = 0; c < nA; ++c) acc += (double)(cm ? Cm[(size_t)c * nT + row] : Cm[(size_t)row * nA + c]) * y[c];
      t[row] = sv[row] - acc;
    }
  }
}

// the whole sequence over nlist elements (list: table positions, or null with a uniform shape);
// max_nA / max_nT: the largest shape (grid extents)
template <typename T>
cudaError_t condense_big(const UnevenArgs& a, const int* list, int nlist, int uni_nA, int uni_nT, int max_nA,
                         int max_nT, cudaStream_t st) {
  if (nlist <= 0) return cudaSuccess;
  if (max_nA > 1024 || max_nT > 16384) return cudaErrorInvalidValue;
  int dev = 0, nsm = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int grid1 = nlist < 4 * nsm ? nlist : 4 * nsm;
  cudaError_t e;
  const size_t psm = lu_panel_smem<T>(max_nA);
  if ((e = cudaFuncSetAttribute(k_big_lu_panel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)psm)) !=
      cudaSuccess)
    return e;
  int occ = 1;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_big_lu_panel<T>, BT, psm)) != cudaSuccess) return e;
  const int gridp = nlist < occ * nsm ? nlist : (occ > 0 ? occ : 1) * nsm;
  (hfr::count_launch(), k_big_lu_init<T><<<grid1, BT, 0, st>>>(a, list, nlist, uni_nA, uni_nT));
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  // one batched GEMM phase over elements [base, base + cnt): rows x cols of the largest shape.  The
  // tensor cores take S = D - C X_B of FP32 blocks (K = nA); the K = 32 updates of the LU, bound by
  // the read-modify-write of their outputs, stay on the CUDA cores
  auto gemm = [&](int base, int cnt, int rows, int cols, int phase, int jb) {
    constexpr int TB = GemmCfg<T>::BM;
    const dim3 g((cols + TB - 1) / TB, (rows + TB - 1) / TB, cnt);
    (hfr::count_launch(), k_big_gemm<T><<<g, BT, 0, st>>>(a, list, base, cnt, uni_nA, uni_nT, phase, jb));
  };
  const int npan = (max_nA + lu_panel<T>() - 1) / lu_panel<T>();
  for (int jb = 0; jb < npan; ++jb) {
    (hfr::count_launch(), k_big_lu_panel<T><<<gridp, BT, psm, st>>>(a, list, nlist, uni_nA, uni_nT, jb));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (jb + 1 == npan) break;
    const int rest = max_nA - (jb + 1) * lu_panel<T>();
    for (int base = 0; base < nlist; base += 65535) {
      const int cnt = nlist - base < 65535 ? nlist - base : 65535;
      gemm(base, cnt, rest, rest, 3, jb);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  // X = A^{-1} P [B | r]: the widest column block whose rows fit shared memory; FP32 blocks of which
  // two CTAs of 64 columns fit an SM (nA up to about 250) take those: one CTA's in-panel solves run
  // under the other's updates (p = 4 and 5 blocks of a wall mesh: 2.0 ms per condensation)
  constexpr int CH = 65535;  // grid y / z extent per launch
  constexpr size_t SM1 = 227 * 1024, SM2 = 113 * 1024;
  auto solve = [&](auto kern, int cw, int nthr, size_t smem, int base, int cnt) -> cudaError_t {
    cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (r != cudaSuccess) return r;
    const dim3 gv((max_nT + 1 + cw - 1) / cw, cnt);  // and the column of r
    (hfr::count_launch(), kern<<<gv, nthr, smem, st>>>(a, list, base, cnt, uni_nA, uni_nT));
    return cudaGetLastError();
  };
  for (int base = 0; base < nlist; base += CH) {
    const int cnt = nlist - base < CH ? nlist - base : CH;
    if constexpr (sizeof(T) == 4) {
      using W = SolveCfg<T, 16, 128, 16, 2>;
      using M = SolveCfg<T, 16, 64, 8, 1>;
      using N = SolveCfg<T, 8, 32, 8, 1>;
      if (M::smem(max_nA) > SM2 && W::smem(max_nA) <= SM1)
        e = solve(k_big_solve<T, 16, 128, 16, 2>, 128, 512, W::smem(max_nA), base, cnt);
      else if (M::smem(max_nA) <= SM1)
        e = solve(k_big_solve<T, 16, 64, 8, 1>, 64, 256, M::smem(max_nA), base, cnt);
      else
        e = solve(k_big_solve<T, 8, 32, 8, 1>, 32, 256, N::smem(max_nA), base, cnt);
    } else {
      using W = SolveCfg<T, 8, 64, 8, 2>;
      using M = SolveCfg<T, 8, 32, 8, 2>;
      using N = SolveCfg<T, 8, 16, 8, 2>;
      if (W::smem(max_nA) <= SM1)
        e = solve(k_big_solve<T, 8, 64, 8, 2>, 64, 256, W::smem(max_nA), base, cnt);
      else if (M::smem(max_nA) <= SM1)
        e = solve(k_big_solve<T, 8, 32, 8, 2>, 32, 256, M::smem(max_nA), base, cnt);
      else
        e = solve(k_big_solve<T, 8, 16, 8, 2>, 16, 256, N::smem(max_nA), base, cnt);
    }
    if (e != cudaSuccess) return e;
    if constexpr (sizeof(T) == 4) {
      auto schur = [&](auto kern, int tm, size_t smem) -> cudaError_t {
        cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (r != cudaSuccess) return r;
        const dim3 g((max_nT + btc::TN - 1) / btc::TN, (max_nT + tm - 1) / tm, cnt);
        (hfr::count_launch(), kern<<<g, btc::THREADS, smem, st>>>(a, list, base, cnt, uni_nA, uni_nT));
        return cudaGetLastError();
      };
      e = max_nT > 128 ? schur(k_big_s_tc<256>, 256, btc::smem<256>()) : schur(k_big_s_tc<128>, 128, btc::smem<128>());
    } else {
      gemm(base, cnt, max_nT, max_nT, 2, 0);
      e = cudaGetLastError();
    }
    if (e != cudaSuccess) return e;
  }
  auto t_kern = k_big_t<T, false>;
  if constexpr (sizeof(T) == 4)
    if (max_nA > XR32_MAX) t_kern = k_big_t<T, true>;
  (hfr::count_launch(), t_kern<<<grid1, BT, 0, st>>>(a, list, nlist, uni_nA, uni_nT));
  return cudaGetLastError();
}

}  // namespace big
}  // namespace hfr
