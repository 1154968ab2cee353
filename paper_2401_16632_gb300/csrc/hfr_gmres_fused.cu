// One restart cycle of right-preconditioned GMRES(m) for the condensed trace system
// L du^ = t (Pereira & Vermeire, arXiv 2401.16632, Sec. 3.2: L = sum_k scatter(S_k) gather_k,
// face-block-Jacobi preconditioner) in a single cooperative launch.
//
// The multi-kernel cycle of hfr_krylov.cu spends most of an iteration launching and draining
// short kernels.  Here one CTA per SM runs the whole cycle: each CTA owns a contiguous range of
// trace faces (and so of every Krylov vector), and the CTAs meet at a grid barrier only where an
// iteration needs data from other faces or a global sum:
//   (A) after z = P^{-1} v_j        (the mat-vec gathers z on neighbouring faces)
//   (B) after w = L z and its dots  (classical Gram-Schmidt coefficients h = V^T w)
//   (C) after w' = w - V h and its dots (second-pass coefficients d = V^T w' and ||w'||)
// Classical Gram-Schmidt is applied twice (CGS2).  The second pass w'' = w' - V d is not a pass
// of its own: its norm follows from ||w''||^2 = ||w'||^2 - ||d||^2 (V orthonormal), and the
// subtraction is folded into the pass that normalises v_{j+1} = w'' / ||w''|| before the next
// preconditioner application.  Only when the second pass removes more than a quarter of
// ||w'||^2 (severe cancellation) is w'' formed and its norm summed explicitly, at one more
// barrier.
// Every CTA reduces the per-CTA partial sums in the same fixed order, so all CTAs hold bitwise
// identical Hessenberg columns, rotations and convergence decisions and take the same path.
// The barrier waits are bounded: a wait that outlasts PG_TIMEOUT_NS raises an abort flag that the
// host reads, and every CTA leaves at its next barrier.
//
// Precision: the Krylov basis, its dots and updates use the block precision T (FP32 in the mixed
// path, where FP64 lanes are 1/64 of the FP32 lanes on this GPU and the GMRES tolerance is loose;
// FP64 in the FP64 path).  The Hessenberg matrix, the Givens rotations, y, the solution du^ and
// the right-hand side stay FP64.  The Givens update of column j-1 (one thread per CTA) runs while
// the other warps finish and precondition v_j, which needs only ||w_j||.
//
// Each CTA reads and writes only its own range of the Krylov vectors, so those accesses go
// through L1; values other CTAs read (z, du^, partial sums) use L2-only loads.  The S blocks,
// re-read by every mat-vec of a cycle, are loaded with an L2 evict-last policy and returned to
// the normal policy when the cycle ends.
#include "hfr_krylov.h"

namespace hfr {

namespace {

constexpr int PG_THREADS = 512;
constexpr int PG_WARPS = PG_THREADS / 32;
constexpr int PG_ND = GM_MAXM + 2;  // dots per reduction: j + 2 <= m + 1
constexpr unsigned long long PG_TIMEOUT_NS = 2000000000ull;
constexpr unsigned PG_MAX_SPINS = 1u << 26;

template <typename T>
struct PGShared {
  T red[PG_ND][PG_WARPS];
  T cf[PG_ND];   // Gram-Schmidt coefficients in the vector precision
  T yT[GM_MAXM];
  T invT;        // 1 / ||w_j||: normalises v_j
  double dot[PG_ND];
  double H[(GM_MAXM + 1) * GM_MAXM];
  double hc[GM_MAXM + 2];
  double g[GM_MAXM + 1];
  double cs[GM_MAXM], sn[GM_MAXM], y[GM_MAXM];
  double rdi[GM_MAXM];  // 1 / H[j][j]
  double beta, bnorm, res, hn;
  int done, k, conv, nan, ok, corr;
};

__device__ __forceinline__ unsigned long long pg_clock() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned pg_load_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Grid barrier of a cooperative launch (all CTAs resident).  bar[0] counts arrivals over the
// whole launch (zeroed before it), bar[1] is the abort flag.  A wait longer than timeout_ns (or
// PG_MAX_SPINS polls) raises the abort flag; a CTA that sees the flag leaves.  Returns false on
// abort.  ok: a shared-memory word of the CTA.
__device__ bool pg_grid_sync(int& ok_shared, unsigned* bar, unsigned& epoch, unsigned long long timeout_ns) {
  __syncthreads();
  ++epoch;
  if (threadIdx.x == 0) {
    int ok = 1;
    const unsigned target = epoch * gridDim.x;
    // release: the CTA's writes (ordered before by the CTA barrier) are visible before the arrival
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    const unsigned long long t0 = pg_clock();
    for (unsigned it = 0; pg_load_acquire(bar) < target; ++it) {
      if ((it & 63u) == 63u) {
        if (pg_load_acquire(bar + 1) != 0u) {
          ok = 0;
          break;
        }
        if (it >= PG_MAX_SPINS || pg_clock() - t0 > timeout_ns) {
          atomicExch(bar + 1, 1u);
          ok = 0;
          break;
        }
      }
      __nanosleep(20);
    }
    ok_shared = ok;
  }
  __syncthreads();
  return ok_shared != 0;
}

template <typename T>
__device__ __forceinline__ bool pg_sync(PGShared<T>& sh, unsigned* bar, unsigned& epoch) {
  return pg_grid_sync(sh.ok, bar, epoch, PG_TIMEOUT_NS);
}

// Self-test of the barrier: `rounds` grid barriers; CTA `absent` (if in range) leaves at once and
// never arrives, so the others' first wait runs out.  passed[0] += barriers each CTA got through.
__global__ void __launch_bounds__(128) k_barrier_probe(unsigned* bar, int absent, int rounds,
                                                       unsigned long long timeout_ns, int* passed) {
  __shared__ int ok;
  if ((int)blockIdx.x == absent) return;
  unsigned epoch = 0;
  int r = 0;
  while (r < rounds && pg_grid_sync(ok, bar, epoch, timeout_ns)) ++r;
  if (threadIdx.x == 0) atomicAdd(passed, r);
}

// Warp reduce-scatter of 16 per-lane values: afterwards lane l holds the warp sum of value l >> 1.
template <typename T>
__device__ __forceinline__ T pg_scatter16(T (&acc)[16], int lane) {
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const bool up = lane & 16;
    const T send = up ? acc[q] : acc[q + 8];
    const T keep = up ? acc[q + 8] : acc[q];
    acc[q] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const bool up = lane & 8;
    const T send = up ? acc[q] : acc[q + 4];
    const T keep = up ? acc[q + 4] : acc[q];
    acc[q] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const bool up = lane & 4;
    const T send = up ? acc[q] : acc[q + 2];
    const T keep = up ? acc[q + 2] : acc[q];
    acc[q] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
  }
  {
    const bool up = lane & 2;
    const T send = up ? acc[0] : acc[1];
    const T keep = up ? acc[1] : acc[0];
    acc[0] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
  }
  return acc[0] + __shfl_xor_sync(0xffffffffu, acc[0], 1);
}

// Warp reduce-scatter of 8 per-lane values: afterwards lane l holds the warp sum of value l >> 2.
template <typename T>
__device__ __forceinline__ T pg_scatter8(T (&acc)[8], int lane) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const bool up = lane & 16;
    const T send = up ? acc[q] : acc[q + 4];
    const T keep = up ? acc[q + 4] : acc[q];
    acc[q] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const bool up = lane & 8;
    const T send = up ? acc[q] : acc[q + 2];
    const T keep = up ? acc[q + 2] : acc[q];
    acc[q] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
  {
    const bool up = lane & 4;
    const T send = up ? acc[0] : acc[1];
    const T keep = up ? acc[1] : acc[0];
    acc[0] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
  }
  acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 2);
  return acc[0] + __shfl_xor_sync(0xffffffffu, acc[0], 1);
}

// 16-byte vector of W values of the basis (W = 16 / sizeof(T)), default (L1-allocating) loads
template <typename T, int W>
struct PGV {
  T v[W];
};
template <typename T, int W>
__device__ __forceinline__ PGV<T, W> pg_ldv(const T* p) {
  PGV<T, W> r;
  if constexpr (sizeof(T) == 4 && W == 4) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    r.v[0] = q.x;
    r.v[1] = q.y;
    r.v[2] = q.z;
    r.v[3] = q.w;
  } else if constexpr (sizeof(T) == 8 && W == 2) {
    const double2 q = *reinterpret_cast<const double2*>(p);
    r.v[0] = q.x;
    r.v[1] = q.y;
  } else {
#pragma unroll
    for (int e = 0; e < W; ++e) r.v[e] = p[e];
  }
  return r;
}
// basis vectors per step of the vector dot pass (two W-vectors of each in flight per thread)
constexpr int PG_VC = 4;
// vector width of the dot pass: 16 bytes when face blocks (hence every CTA's range and the vector
// length) are whole vectors, else scalar
template <typename T, int BS>
__host__ __device__ constexpr int pg_basis_width() {
  return BS % (16 / (int)sizeof(T)) == 0 ? 16 / (int)sizeof(T) : 1;
}

// The FP64 form of the dot pass below.  Every FP64 instruction of a warp occupies the SM's FP64 pipe
// for about 19 cycles, whatever its lanes hold, so the pass spends them on products alone: one
// multiply-add per value and basis vector (sixteen vectors at a time, their loads in flight
// together), a lane reduction sized to the vectors left, and none in warps without entries.  The
// paired form that FP32 uses cost half as many again in separate products, and as many lanes of the
// last step (459 000 values, 16 vectors: 40 us against 25).  Entries are visited as the updates of this file do.
__device__ __forceinline__ double pg_lane_sum16(double (&acc)[16], int cnt, int lane) {
  // butterfly over the lane bits 4 .. 1 (each level halves the values a lane carries), then bit 0:
  // lane l ends with the warp sum of value l >> 1; levels whose upper half is empty only add
  double v8[8], v4[4], v2[2];
  const bool u4 = lane & 16, u3 = lane & 8, u2 = lane & 4, u1 = lane & 2;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const double send = u4 ? acc[q] : acc[q + 8], keep = u4 ? acc[q + 8] : acc[q];
    v8[q] = q < cnt ? keep + __shfl_xor_sync(0xffffffffu, send, 16) : 0.0;
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const double send = u3 ? v8[q] : v8[q + 4], keep = u3 ? v8[q + 4] : v8[q];
    v4[q] = q < cnt ? keep + __shfl_xor_sync(0xffffffffu, send, 8) : 0.0;
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const double send = u2 ? v4[q] : v4[q + 2], keep = u2 ? v4[q + 2] : v4[q];
    v2[q] = q < cnt ? keep + __shfl_xor_sync(0xffffffffu, send, 4) : 0.0;
  }
  const double send = u1 ? v2[0] : v2[1], keep = u1 ? v2[1] : v2[0];
  const double r = keep + __shfl_xor_sync(0xffffffffu, send, 2);
  return r + __shfl_xor_sync(0xffffffffu, r, 1);
}
__device__ void pg_block_dots64(PGShared<double>& sh, const double* V, size_t n, int nd, const double* w, size_t x0,
                                size_t x1, double* partial) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const size_t nw = (x1 - x0 + 31) / 32;
  const int active = nw < PG_WARPS ? (int)nw : PG_WARPS;  // warps with entries
  if (wid < active) {
    for (int c0 = 0; c0 < nd; c0 += 16) {
      const int cnt = min(16, nd - c0);
      double acc[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) acc[q] = 0.0;
      for (size_t x = x0 + threadIdx.x; x < x1; x += PG_THREADS) {
        const double wx = w[x];
        double v[16];
#pragma unroll
        for (int q = 0; q < 16; ++q)
          if (q < cnt) v[q] = V[(size_t)(c0 + q) * n + x];
#pragma unroll
        for (int q = 0; q < 16; ++q)
          if (q < cnt) acc[q] = fma(v[q], wx, acc[q]);
      }
      const double s = pg_lane_sum16(acc, cnt, lane);
      const int vi = c0 + (lane >> 1);
      if ((lane & 1) == 0 && vi < nd) sh.red[vi][wid] = s;
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nd; i += PG_THREADS) {
    double t = 0.0;
    for (int k = 0; k < active; ++k) t += sh.red[i][k];
    partial[(size_t)i * gridDim.x + blockIdx.x] = t;
  }
}

// CTA partial of V_i . w over this CTA's entries [x0, x1), i < nd, written to
// partial[i * gridDim.x + blockIdx.x].  Each thread visits the entries x0 + tid + PG_THREADS u,
// the same ones the vector updates of this file give it, so it only re-reads its own writes.
// With W > 1 the thread visits the W-vectors x0 / W + tid + PG_THREADS u instead (two W-vectors of
// w and of PG_VC basis vectors per step, 2 PG_VC + 2 loads of 16 bytes in flight); w's entries are
// then not the thread's own writes, so the caller puts a block barrier between the update of w and
// this pass.
template <typename T, int W = 1>
__device__ void pg_block_dots(PGShared<T>& sh, const T* V, size_t n, int nd, const T* w, size_t x0, size_t x1,
                              T* partial) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if constexpr (sizeof(T) == 8) {
    pg_block_dots64(sh, V, n, nd, w, x0, x1, partial);
  } else if constexpr (W > 1) {
    const size_t g0 = x0 / W, g1 = x1 / W, nW = n / W;
    for (int c0 = 0; c0 < nd; c0 += PG_VC) {
      T acc[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) acc[q] = T(0);
      for (size_t ga = g0 + threadIdx.x; ga < g1; ga += 2 * PG_THREADS) {
        const size_t gb = ga + PG_THREADS;
        const bool okb = gb < g1;
        const size_t gbs = okb ? gb : ga;
        const PGV<T, W> wa = pg_ldv<T, W>(w + ga * W);
        PGV<T, W> wb = pg_ldv<T, W>(w + gbs * W);
        if (!okb) {
#pragma unroll
          for (int e = 0; e < W; ++e) wb.v[e] = T(0);
        }
        PGV<T, W> va[PG_VC], vb[PG_VC];
#pragma unroll
        for (int q = 0; q < PG_VC; ++q)
          if (c0 + q < nd) {
            va[q] = pg_ldv<T, W>(V + ((size_t)(c0 + q) * nW + ga) * W);
            vb[q] = pg_ldv<T, W>(V + ((size_t)(c0 + q) * nW + gbs) * W);
          }
#pragma unroll
        for (int q = 0; q < PG_VC; ++q)
          if (c0 + q < nd) {
#pragma unroll
            for (int e = 0; e < W; ++e) acc[q] += va[q].v[e] * wa.v[e] + vb[q].v[e] * wb.v[e];
          }
      }
      const T s = pg_scatter8(acc, lane);
      const int vi = c0 + (lane >> 2);
      if ((lane & 3) == 0 && vi < nd) sh.red[vi][wid] = s;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nd; i += PG_THREADS) {
      T t = T(0);
#pragma unroll
      for (int k = 0; k < PG_WARPS; ++k) t += sh.red[i][k];
      partial[(size_t)i * gridDim.x + blockIdx.x] = t;
    }
  } else {
    for (int c0 = 0; c0 < nd; c0 += 16) {
      T acc[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) acc[q] = T(0);
      // two entries per iteration: 34 independent loads in flight per thread
      for (size_t xa = x0 + threadIdx.x; xa < x1; xa += 2 * PG_THREADS) {
        const size_t xb = xa + PG_THREADS;
        const bool okb = xb < x1;
        const T wa = w[xa];
        const T wb = okb ? w[xb] : T(0);
        const size_t xbs = okb ? xb : xa;
#pragma unroll
        for (int q = 0; q < 16; ++q)
          if (c0 + q < nd) {
            const T va = V[(size_t)(c0 + q) * n + xa];
            const T vb = V[(size_t)(c0 + q) * n + xbs];
            acc[q] += va * wa + vb * wb;
          }
      }
      const T s = pg_scatter16(acc, lane);
      const int vi = c0 + (lane >> 1);
      if ((lane & 1) == 0 && vi < nd) sh.red[vi][wid] = s;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nd; i += PG_THREADS) {
      T t = T(0);
#pragma unroll
      for (int k = 0; k < PG_WARPS; ++k) t += sh.red[i][k];
      partial[(size_t)i * gridDim.x + blockIdx.x] = t;
    }
  }
}

// CTA partials of ||u||^2 (slot 0) and, if v, ||v||^2 (slot 1), in the vector precision
template <typename T, typename U2>
__device__ void pg_block_sq(PGShared<T>& sh, const T* u, const U2* v, size_t x0, size_t x1, T* partial) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  T su = T(0), sv = T(0);
  for (size_t x = x0 + threadIdx.x; x < x1; x += PG_THREADS) {
    const T a = u[x];
    su += a * a;
    if (v) {
      const T b = T(__ldcg(v + x));
      sv += b * b;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    su += __shfl_xor_sync(0xffffffffu, su, o);
    sv += __shfl_xor_sync(0xffffffffu, sv, o);
  }
  if (lane == 0) {
    sh.red[0][wid] = su;
    sh.red[1][wid] = sv;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    T t = T(0);
#pragma unroll
    for (int k = 0; k < PG_WARPS; ++k) t += sh.red[threadIdx.x][k];
    partial[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = t;
  }
}

// After the barrier: sh.dot[i] = sum over CTAs of partial slot i, in the same order everywhere.
template <typename T>
__device__ void pg_reduce(PGShared<T>& sh, int nd, const T* partial) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nb = (int)gridDim.x;
  for (int i = wid; i < nd; i += PG_WARPS) {
    const T* pi = partial + (size_t)i * nb;
    T t = T(0);
    for (int b0 = 0; b0 < nb; b0 += 32 * 8) {
      T v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int b = b0 + lane + 32 * q;
        v[q] = b < nb ? __ldcg(pi + b) : T(0);
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) t += v[q];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) sh.dot[i] = double(t);
  }
  __syncthreads();
}

// Vector loads of VW consecutive values.  The S blocks are read with an L2 evict-last policy so
// that they stay resident in L2 across the iterations of a cycle (they are the largest operand and
// are re-read by every mat-vec); everything else uses the default policy.
template <typename T, int VW>
struct PGVec {
  T v[VW];
};

__device__ __forceinline__ unsigned long long pg_policy_keep() {
  unsigned long long p;
  asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}

template <typename T, int VW>
__device__ __forceinline__ PGVec<T, VW> pg_ld_keep(const T* ptr, unsigned long long pol) {
  PGVec<T, VW> r;
  if constexpr (sizeof(T) == 4 && VW == 4) {
    asm("ld.global.nc.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
        : "=f"(r.v[0]), "=f"(r.v[1]), "=f"(r.v[2]), "=f"(r.v[3])
        : "l"(ptr), "l"(pol));
  } else if constexpr (sizeof(T) == 4 && VW == 2) {
    asm("ld.global.nc.L2::cache_hint.v2.f32 {%0, %1}, [%2], %3;" : "=f"(r.v[0]), "=f"(r.v[1]) : "l"(ptr), "l"(pol));
  } else if constexpr (sizeof(T) == 8 && VW == 2) {
    asm("ld.global.nc.L2::cache_hint.v2.f64 {%0, %1}, [%2], %3;" : "=d"(r.v[0]), "=d"(r.v[1]) : "l"(ptr), "l"(pol));
  } else {
#pragma unroll
    for (int q = 0; q < VW; ++q) r.v[q] = __ldg(ptr + q);
  }
  return r;
}

// VW consecutive BF16 values (the trace operator stored in BF16) widened to FP32, with the same
// evict-last policy; BF16 is the upper half of an FP32 word, so widening is a 16-bit shift
template <int VW>
__device__ __forceinline__ PGVec<float, VW> pg_ld_keep_bf16(const unsigned short* ptr, unsigned long long pol) {
  PGVec<float, VW> r;
  if constexpr (VW == 4) {
    unsigned a, b;
    asm("ld.global.nc.L2::cache_hint.v2.u32 {%0, %1}, [%2], %3;" : "=r"(a), "=r"(b) : "l"(ptr), "l"(pol));
    r.v[0] = __uint_as_float(a << 16);
    r.v[1] = __uint_as_float(a & 0xffff0000u);
    r.v[2] = __uint_as_float(b << 16);
    r.v[3] = __uint_as_float(b & 0xffff0000u);
  } else if constexpr (VW == 2) {
    unsigned a;
    asm("ld.global.nc.L2::cache_hint.u32 %0, [%1], %2;" : "=r"(a) : "l"(ptr), "l"(pol));
    r.v[0] = __uint_as_float(a << 16);
    r.v[1] = __uint_as_float(a & 0xffff0000u);
  } else {
#pragma unroll
    for (int q = 0; q < VW; ++q) r.v[q] = __uint_as_float((unsigned)__ldg(ptr + q) << 16);
  }
  return r;
}

template <typename T, int VW>
__device__ __forceinline__ PGVec<T, VW> pg_ld_cg(const T* ptr) {
  PGVec<T, VW> r;
  if constexpr (sizeof(T) == 4 && VW == 4) {
    const float4 q = __ldcg(reinterpret_cast<const float4*>(ptr));
    r.v[0] = q.x;
    r.v[1] = q.y;
    r.v[2] = q.z;
    r.v[3] = q.w;
  } else if constexpr (sizeof(T) == 4 && VW == 2) {
    const float2 q = __ldcg(reinterpret_cast<const float2*>(ptr));
    r.v[0] = q.x;
    r.v[1] = q.y;
  } else if constexpr (sizeof(T) == 8 && VW == 2) {
    const double2 q = __ldcg(reinterpret_cast<const double2*>(ptr));
    r.v[0] = q.x;
    r.v[1] = q.y;
  } else {
#pragma unroll
    for (int q = 0; q < VW; ++q) r.v[q] = __ldcg(ptr + q);
  }
  return r;
}

// VW consecutive values that are not written during the kernel (16-byte vectors)
template <typename T, int VW>
__device__ __forceinline__ PGVec<T, VW> pg_ld_stream(const T* ptr) {
  PGVec<T, VW> r;
  if constexpr (sizeof(T) == 4) {
    const float4 q = __ldg(reinterpret_cast<const float4*>(ptr));
    r.v[0] = q.x;
    r.v[1] = q.y;
    r.v[2] = q.z;
    r.v[3] = q.w;
  } else {
    const double2 q = __ldg(reinterpret_cast<const double2*>(ptr));
    r.v[0] = q.x;
    r.v[1] = q.y;
  }
  return r;
}

// widest vector (16 bytes at most) that divides both the per-lane column count and the face block
template <typename T, int NT, int BS>
struct PGShape {
  static constexpr int CT = NT / 8;  // columns per lane
  static constexpr int VMAX = 16 / (int)sizeof(T);
  static constexpr int VW = (CT % 4 == 0 && BS % 4 == 0 && VMAX >= 4) ? 4 : ((CT % 2 == 0 && BS % 2 == 0) ? 2 : 1);
  static constexpr int CV = CT / VW;  // vectors per lane and row
  static constexpr int RU = (BS + 3) / 4;
  static_assert(NT % 8 == 0, "nT must be a multiple of 8");
};

// Rows grp + 4u of (L s)_f for trace face f, in every lane of 8-lane group grp: both neighbours'
// row blocks of S_k against the neighbours' gathered trace values (src in the block precision T,
// or FP64 when SRC_D).  Lane g8 of a group holds the columns VW (g8 + 8 c) + q of each row, so
// every load is a VW-wide vector and no vector crosses a face block.
template <typename T, int NT, int BS, bool SRC_D, bool SB>
__device__ __forceinline__ void pg_face_rows(const FusedArgs& a, int f, const void* src, unsigned long long pol,
                                             T (&acc)[(BS + 3) / 4]) {
  using Sh = PGShape<T, NT, BS>;
  constexpr int VW = Sh::VW, CV = Sh::CV, RU = Sh::RU;
  // both sides' rows in flight at once when they fit in registers
  constexpr bool BOTH = 2 * RU * CV * VW * (int)sizeof(T) <= 256;
  const int lane = threadIdx.x & 31;
  const int grp = lane >> 3, g8 = lane & 7;
  const T* S = reinterpret_cast<const T*>(a.S);
#pragma unroll
  for (int u = 0; u < RU; ++u) acc[u] = T(0);
#pragma unroll(BOTH ? 2 : 1)
  for (int side = 0; side < 2; ++side) {
    const int e = __ldg(a.sides + f * 4 + side * 2);
    if (e < 0) continue;
    const int fs = __ldg(a.sides + f * 4 + side * 2 + 1);
    PGVec<T, VW> sv[RU][CV];
#pragma unroll
    for (int u = 0; u < RU; ++u) {
      const int i = grp + 4 * u;
      const int ii = i < BS ? i : 0;
      const size_t ro = ((size_t)e * NT + (size_t)fs * BS + ii) * NT;
      if constexpr (SB) {
        const unsigned short* row = reinterpret_cast<const unsigned short*>(a.S) + ro;
#pragma unroll
        for (int c = 0; c < CV; ++c) {
          const PGVec<float, VW> x = pg_ld_keep_bf16<VW>(row + VW * (g8 + 8 * c), pol);
#pragma unroll
          for (int q = 0; q < VW; ++q) sv[u][c].v[q] = T(x.v[q]);
        }
      } else {
        const T* row = S + ro;
#pragma unroll
        for (int c = 0; c < CV; ++c) sv[u][c] = pg_ld_keep<T, VW>(row + VW * (g8 + 8 * c), pol);
      }
    }
    PGVec<T, VW> xv[CV];
#pragma unroll
    for (int c = 0; c < CV; ++c) {
      const int l = VW * (g8 + 8 * c);
      const int fp = l / BS;
      const int tf = __ldg(a.tr_of_c + e * 4 + fp);
      const size_t ix = (size_t)(tf >= 0 ? tf : 0) * BS + (l - fp * BS);
      if (SRC_D) {
        const PGVec<double, VW> d = pg_ld_cg<double, VW>(reinterpret_cast<const double*>(src) + ix);
#pragma unroll
        for (int q = 0; q < VW; ++q) xv[c].v[q] = tf >= 0 ? T(d.v[q]) : T(0);
      } else {
        xv[c] = pg_ld_cg<T, VW>(reinterpret_cast<const T*>(src) + ix);
        if (tf < 0) {
#pragma unroll
          for (int q = 0; q < VW; ++q) xv[c].v[q] = T(0);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < RU; ++u) {
      if (grp + 4 * u < BS) {
#pragma unroll
        for (int c = 0; c < CV; ++c)
#pragma unroll
          for (int q = 0; q < VW; ++q) acc[u] += sv[u][c].v[q] * xv[c].v[q];
      }
    }
  }
#pragma unroll
  for (int u = 0; u < RU; ++u) {
    acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], 4);
    acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], 2);
    acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], 1);
  }
}

// out_f = t_f - (L src)_f when RES, else (L src)_f, for this CTA's faces (one warp per face),
// stored in the vector precision T
template <typename T, int NT, int BS, bool SRC_D, bool RES, bool SB>
__device__ void pg_matvec(const FusedArgs& a, const void* src, T* out, int fb0, int fb1) {
  constexpr int RU = (BS + 3) / 4;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int grp = lane >> 3, g8 = lane & 7;
  const unsigned long long pol = pg_policy_keep();
  for (int f = fb0 + wid; f < fb1; f += PG_WARPS) {
    T acc[RU];
    pg_face_rows<T, NT, BS, SRC_D, SB>(a, f, src, pol, acc);
    if (g8 == 0) {
#pragma unroll
      for (int u = 0; u < RU; ++u) {
        const int i = grp + 4 * u;
        if (i < BS) {
          const size_t ix = (size_t)f * BS + i;
          out[ix] = RES ? T(__ldcg(a.t + ix) - double(acc[u])) : acc[u];
        }
      }
    }
  }
}

// Row r of the face block P_f^{-1} (block precision) into registers
template <typename T, int BS>
__device__ __forceinline__ void pg_prow(const T* P, int f, int r, T (&row)[BS]) {
  const T* src = P + ((size_t)f * BS + r) * BS;
  if constexpr (sizeof(T) == 4 && BS % 4 == 0) {
#pragma unroll
    for (int c = 0; c < BS / 4; ++c) {
      const float4 q = __ldg(reinterpret_cast<const float4*>(src) + c);
      row[4 * c] = q.x;
      row[4 * c + 1] = q.y;
      row[4 * c + 2] = q.z;
      row[4 * c + 3] = q.w;
    }
  } else {
#pragma unroll
    for (int c = 0; c < BS; ++c) row[c] = __ldg(src + c);
  }
}

// z = P^{-1} v_j, one warp per face of this CTA (two faces per step), lane r < BS owns row r.
// Warp 0 takes no face: its lane 0 updates the Givens rotations meanwhile.
template <typename T, int BS>
__device__ void pg_precond(const FusedArgs& a, const T* vj, int fb0, int fb1) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (wid == 0) return;
  const T* P = reinterpret_cast<const T*>(a.Pinv);
  T* z = reinterpret_cast<T*>(a.z);
  const int r = lane < BS ? lane : 0;
  constexpr int NW = PG_WARPS - 1;
  for (int f = fb0 + wid - 1; f < fb1; f += 2 * NW) {
    // two faces per step: both blocks' loads in flight together
    const int f2 = f + NW;
    const bool two = f2 < fb1;
    const size_t ix = (size_t)f * BS + r, ix2 = (size_t)(two ? f2 : f) * BS + r;
    const T v = lane < BS ? vj[ix] : T(0);
    const T v2 = lane < BS ? vj[ix2] : T(0);
    T row[BS], row2[BS];
    pg_prow<T, BS>(P, f, r, row);
    pg_prow<T, BS>(P, two ? f2 : f, r, row2);
    T acc = T(0), acc2 = T(0);
#pragma unroll
    for (int c = 0; c < BS; ++c) {
      acc += row[c] * __shfl_sync(0xffffffffu, v, c);
      acc2 += row2[c] * __shfl_sync(0xffffffffu, v2, c);
    }
    if (lane < BS) {
      z[ix] = acc;
      if (two) z[ix2] = acc2;
    }
  }
}

// dst[x] = (dst[x] - sum_{i<cnt} c_i V_i[x]) * scale over the entries x0 + tid0 + m nthreads of this
// thread; four entries per iteration and two basis vectors per inner step keep eight independent
// loads in flight per thread (the basis of a large system streams from HBM)
template <typename T>
__device__ __forceinline__ void pg_axpy_multi(const T* V, size_t n, const T* c, int cnt, T* dst, T scale,
                                              size_t x0, size_t x1, int tid0, int nthreads) {
  const size_t st = (size_t)nthreads;
  if constexpr (sizeof(T) == 8) {  // one multiply-add per value and vector (see the FP64 dot pass)
    for (size_t x = x0 + tid0; x < x1; x += st) {
      T s0 = T(0), s1 = T(0);
      int i = 0;
      for (; i + 8 <= cnt; i += 8) {
        T v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = V[(size_t)(i + u) * n + x];
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
          s0 = fma(c[i + u], v[u], s0);
          s1 = fma(c[i + u + 1], v[u + 1], s1);
        }
      }
      for (; i < cnt; ++i) s0 = fma(c[i], V[(size_t)i * n + x], s0);
      dst[x] = (dst[x] - (s0 + s1)) * scale;
    }
  } else {
  for (size_t xb = x0 + tid0; xb < x1; xb += 4 * st) {
    size_t xs[4];
    bool ok[4];
    T sacc[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      xs[u] = xb + u * st;
      ok[u] = xs[u] < x1;
      if (!ok[u]) xs[u] = xb;
      sacc[u] = T(0);
    }
    int i = 0;
    for (; i + 2 <= cnt; i += 2) {
      const T ca = c[i], cb = c[i + 1];
      const T* Va = V + (size_t)i * n;
      const T* Vb = Va + n;
#pragma unroll
      for (int u = 0; u < 4; ++u) sacc[u] += ca * Va[xs[u]] + cb * Vb[xs[u]];
    }
    if (i < cnt) {
      const T ca = c[i];
      const T* Va = V + (size_t)i * n;
#pragma unroll
      for (int u = 0; u < 4; ++u) sacc[u] += ca * Va[xs[u]];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (ok[u]) dst[xs[u]] = (dst[xs[u]] - sacc[u]) * scale;
  }
  }
}

// v_j <- (v_j - sum_{i<jc} c_i V_i) * inv over this CTA's entries, by warps 1.. only (jc = 0: scale)
template <typename T>
__device__ void pg_finish(const T* V, size_t n, const T* c, int jc, T inv, T* vj, size_t x0, size_t x1) {
  if (threadIdx.x < 32) return;
  pg_axpy_multi(V, n, c, jc, vj, inv, x0, x1, (int)threadIdx.x - 32, PG_THREADS - 32);
}

// named barrier of warps 1 .. PG_WARPS-1 (warp 0 is busy with the Givens update)
__device__ __forceinline__ void pg_sync_workers() {
  asm volatile("bar.sync 1, %0;" ::"n"(PG_THREADS - 32) : "memory");
}

// x_f += P_f^{-1} (sum_{i<k} y_i V_i)_f: first u = V y over this CTA's entries into the z buffer
// (free at the end of the cycle; a streaming pass with many loads in flight), then P_f^{-1} u_f in
// the vector precision added to the FP64 solution, one warp per face
template <typename T, int BS>
__device__ void pg_update_x(const FusedArgs& a, const PGShared<T>& sh, const T* V, int k, int fb0, int fb1) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const T* P = reinterpret_cast<const T*>(a.Pinv);
  T* u = reinterpret_cast<T*>(a.z);
  const size_t x0 = (size_t)fb0 * BS, x1 = (size_t)fb1 * BS;
  for (size_t x = x0 + threadIdx.x; x < x1; x += PG_THREADS) u[x] = T(0);
  __syncthreads();
  pg_axpy_multi(V, a.n, sh.yT, k, u, T(-1), x0, x1, (int)threadIdx.x, PG_THREADS);
  __syncthreads();
  const int r = lane < BS ? lane : 0;
  for (int f = fb0 + wid; f < fb1; f += PG_WARPS) {
    const size_t ix = (size_t)f * BS + r;
    const T uv = lane < BS ? u[ix] : T(0);
    T row[BS];
    pg_prow<T, BS>(P, f, r, row);
    T acc = T(0);
#pragma unroll
    for (int c = 0; c < BS; ++c) acc += row[c] * __shfl_sync(0xffffffffu, uv, c);
    if (lane < BS) a.x[ix] += double(acc);
  }
}

template <typename T>
__device__ __forceinline__ void pg_subtract(const T* V, size_t n, const T* c, int j, T* w, size_t x0, size_t x1) {
  pg_axpy_multi(V, n, c, j + 1, w, T(1), x0, x1, (int)threadIdx.x, PG_THREADS);
}

// Givens update of Hessenberg column j (sh.hc[0..j+1]), FP64; decides the end of the cycle
template <typename T>
__device__ void pg_givens(PGShared<T>& sh, int j, double rtol, int m) {
  double* h = sh.hc;
  for (int i = 0; i < j; ++i) {
    const double a = h[i], b = h[i + 1];
    h[i] = sh.cs[i] * a + sh.sn[i] * b;
    h[i + 1] = -sh.sn[i] * a + sh.cs[i] * b;
  }
  const double a = h[j], b = h[j + 1];
  sh.hn = b;
  const double r = sqrt(a * a + b * b);
  const double ri = r > 0.0 ? 1.0 / r : 0.0;
  double c = 1.0, s = 0.0;
  if (r > 0.0) {
    c = a * ri;
    s = b * ri;
  }
  sh.cs[j] = c;
  sh.sn[j] = s;
  sh.rdi[j] = ri;
  h[j] = r;
  for (int i = 0; i <= j; ++i) sh.H[i * GM_MAXM + j] = h[i];
  sh.g[j + 1] = -s * sh.g[j];
  sh.g[j] = c * sh.g[j];
  sh.res = fabs(sh.g[j + 1]);
  sh.k = j + 1;
  if (!(sh.res == sh.res)) {
    sh.nan = 1;
    sh.done = 1;
  } else if (sh.res <= rtol * sh.bnorm) {
    sh.conv = 1;
    sh.done = 1;
  } else if (j + 1 >= m || b == 0.0) {
    sh.done = 1;
  }
}

template <typename T, int NT, int BS, bool SB>
__global__ void __launch_bounds__(PG_THREADS, 1) k_gmres_cycle(const __grid_constant__ FusedArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PGShared<T>& sh = *reinterpret_cast<PGShared<T>*>(smem_raw);
  const int F = a.ntrace;
  const int fb0 = (int)((long long)blockIdx.x * F / gridDim.x);
  const int fb1 = (int)((long long)(blockIdx.x + 1) * F / gridDim.x);
  const size_t n = a.n, x0 = (size_t)fb0 * BS, x1 = (size_t)fb1 * BS;
  constexpr int VWB = pg_basis_width<T, BS>();
  const int tid = threadIdx.x;
  unsigned epoch = 0;
  int par = 0;
  const size_t pstride = (size_t)PG_ND * gridDim.x;
  T* V = reinterpret_cast<T*>(a.V);
  T* const partial = reinterpret_cast<T*>(a.partial);

  const int xz = a.dyn ? a.dyn[0] : a.x_zero;
  const int mm = a.dyn ? a.dyn[1] : a.m;
  // r0 = t - L x into V_0 (x = 0: r0 = t); beta = ||r0||, bnorm = ||t||
  if (xz) {
    for (size_t x = x0 + tid; x < x1; x += PG_THREADS) V[x] = T(__ldcg(a.t + x));
  } else {
    pg_matvec<T, NT, BS, true, true, SB>(a, a.x, V, fb0, fb1);
  }
  __syncthreads();
  pg_block_sq(sh, V, a.t, x0, x1, partial + par * pstride);
  if (!pg_sync(sh, a.bar, epoch)) return;
  pg_reduce(sh, 2, partial + par * pstride);
  par ^= 1;
  if (tid == 0) {
    const double beta = sqrt(sh.dot[0]);
    sh.beta = beta;
    sh.bnorm = sqrt(sh.dot[1]);
    sh.g[0] = beta;
    sh.res = beta;
    sh.hn = beta;
    sh.k = 0;
    sh.conv = 0;
    sh.nan = 0;
    sh.done = 0;
    sh.corr = 0;
    sh.invT = T(beta > 0.0 ? 1.0 / beta : 0.0);
    if (!(beta == beta)) {
      sh.nan = 1;
      sh.done = 1;
    } else if (beta <= a.rtol * sh.bnorm || beta == 0.0) {
      sh.conv = 1;
      sh.done = 1;
    }
  }
  __syncthreads();

  if (!sh.done) {
    for (int j = 0;; ++j) {
      T* vj = V + (size_t)j * n;
      T* w = V + (size_t)(j + 1) * n;
      // (A) lane 0 of warp 0: Givens rotation of column j-1.  Warps 1..: finish v_j (deferred
      // second Gram-Schmidt pass, normalisation) and form z = P^{-1} v_j.
      if (j > 0 && tid == 0) pg_givens(sh, j - 1, a.rtol, mm);
      if (tid >= 32) {
        pg_finish(V, n, sh.cf, sh.corr ? j : 0, sh.invT, vj, x0, x1);
        pg_sync_workers();
        pg_precond<T, BS>(a, vj, fb0, fb1);
      }
      if (!pg_sync(sh, a.bar, epoch)) return;
      if (sh.done) break;
      // (B) w = L z and h = V^T w
      pg_matvec<T, NT, BS, false, false, SB>(a, a.z, w, fb0, fb1);
      __syncthreads();
      T* part = partial + par * pstride;
      pg_block_dots<T, VWB>(sh, V, n, j + 1, w, x0, x1, part);
      if (!pg_sync(sh, a.bar, epoch)) return;
      pg_reduce(sh, j + 1, part);
      par ^= 1;
      for (int i = tid; i <= j; i += PG_THREADS) {
        sh.hc[i] = sh.dot[i];
        sh.cf[i] = T(sh.dot[i]);
      }
      __syncthreads();
      // (C) w' = w - V h, then d = V^T w' and ||w'||^2 (dot j+1: V_{j+1} is w' itself)
      pg_subtract(V, n, sh.cf, j, w, x0, x1);
      if (VWB > 1) __syncthreads();  // the dot pass visits w in its own (vector) order
      part = partial + par * pstride;
      pg_block_dots<T, VWB>(sh, V, n, j + 2, w, x0, x1, part);
      if (!pg_sync(sh, a.bar, epoch)) return;
      pg_reduce(sh, j + 2, part);
      par ^= 1;
      if (tid < 32) {
        // ||d||^2 (fixed order), h += d, coefficients of the deferred pass
        double dd = 0.0;
        for (int i = tid; i <= j; i += 32) {
          const double d = sh.dot[i];
          dd += d * d;
          sh.hc[i] += d;
          sh.cf[i] = T(d);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) dd += __shfl_xor_sync(0xffffffffu, dd, o);
        if (tid == 0) {
          const double n1 = sh.dot[j + 1];
          sh.corr = dd <= 0.25 * n1 ? 1 : 0;
          if (sh.corr) sh.hc[j + 1] = sqrt(n1 - dd);
        }
      }
      __syncthreads();
      if (!sh.corr) {
        // severe cancellation: form w'' = w' - V d now and sum its norm
        pg_subtract(V, n, sh.cf, j, w, x0, x1);
        part = partial + par * pstride;
        pg_block_sq(sh, w, (const T*)nullptr, x0, x1, part);
        if (!pg_sync(sh, a.bar, epoch)) return;
        pg_reduce(sh, 1, part);
        par ^= 1;
        if (tid == 0) sh.hc[j + 1] = sqrt(sh.dot[0]);
      }
      if (tid == 0) sh.invT = T(sh.hc[j + 1] != 0.0 ? 1.0 / sh.hc[j + 1] : 0.0);
      __syncthreads();
    }
  }

  // y = H^{-1} g, x += P^{-1} V y
  const int k = sh.k;
  if (tid == 0) {
    for (int i = k - 1; i >= 0; --i) {
      double s = sh.g[i];
      for (int c = i + 1; c < k; ++c) s -= sh.H[i * GM_MAXM + c] * sh.y[c];
      sh.y[i] = s * sh.rdi[i];
      sh.yT[i] = T(sh.y[i]);
    }
  }
  __syncthreads();
  if (k > 0) pg_update_x<T, BS>(a, sh, V, k, fb0, fb1);
  if (a.true_res) {
    // true residual ||t - L x|| (V_0 as scratch)
    if (!pg_sync(sh, a.bar, epoch)) return;
    pg_matvec<T, NT, BS, true, true, SB>(a, a.x, V, fb0, fb1);
    __syncthreads();
    pg_block_sq(sh, V, (const T*)nullptr, x0, x1, partial + par * pstride);
    if (!pg_sync(sh, a.bar, epoch)) return;
    pg_reduce(sh, 1, partial + par * pstride);
  }
  // the S blocks go back to the normal L2 eviction policy (the next condensation rewrites them)
  for (size_t off = ((size_t)blockIdx.x * PG_THREADS + tid) * 128; off < a.S_bytes;
       off += (size_t)gridDim.x * PG_THREADS * 128)
    asm volatile("applypriority.global.L2::evict_normal [%0], 128;" ::"l"(reinterpret_cast<const char*>(a.S) + off)
                 : "memory");
  if (blockIdx.x == 0 && tid == 0) {
    GmresState* st = a.st;
    st->beta = a.true_res ? sqrt(sh.dot[0]) : sh.res;
    st->bnorm = sh.bnorm;
    st->res = sh.res;
    st->hn = sh.hn;
    st->k = k;
    st->kdone = k;
    st->converged = sh.conv;
    st->nan = sh.nan;
  }
}

// ------------------------------------------------------- the cycle on any trace layout
// The same iteration with an FP64 basis, for trace units of any size and element blocks of any shape
// (mixed degrees, hexahedra, EFR nodes, uniform shapes without a compiled cycle).  The operator runs
// in the element view, which adds one barrier: (A) z = P^-1 v_j; (B) y_k = S_k z_k; (C) w = the sum of
// the element entries, h = V^T w; (D) w' = w - V h, d = V^T w', ||w'||.  Z keeps P^-1 v_j, so x
// moves by sum y_j z_j with the very vectors that the operator saw.
//
// What bounds it: the S blocks from HBM in (B), the FP64 pipe in (C), (D) and the deferred second
// pass (4 (j + 1) n multiply-adds per iteration).  The S values are cut into equal runs of rows, one
// per warp of the grid, whatever the element shapes.  As one kernel per step (seven launches per
// iteration, two of them reductions that ended in one block reading every partial sum and updating
// the rotations from global memory) an iteration of a stage costs 284 us on EFR nodes (128 x 128, p = 4),
// 297 us on a wall mesh of 10 000 implicit elements and 70 us on 64 scalar elements; it takes 245, 203
// and 26 us here.
// Systems of some hundred values run on one cluster of eight CTAs, whose barrier is hardware.

struct AnyShape {  // the layout of one element or trace unit, from the tables or the uniform sizes
  const CycleArgs& a;
  __device__ __forceinline__ int nT(int k) const { return a.uni_nT ? a.uni_nT : __ldg(a.nTk + k); }
  __device__ __forceinline__ long long offD(int k) const {
    return a.uni_nT ? (long long)k * a.uni_nT * a.uni_nT : __ldg(a.offD + k);
  }
  __device__ __forceinline__ long long offs(int k) const {
    return a.uni_nT ? (long long)k * a.uni_nT : __ldg(a.offs + k);
  }
  // trace value of local unknown l of element k (its entries start at o), -1 off traces
  __device__ __forceinline__ long long gmap(int k, long long o, int l) const {
    if (!a.uni_nT) {
      const int g = __ldg(a.gmap + o + l);
      return g < 0 ? -1 : (long long)FR_IDX(g, a.n, 31);
    }
    const int f = l / a.uni_bs, t = __ldg(a.tr_of_c + 4 * k + f);
    return t < 0 ? -1 : (long long)FR_IDX(t, a.ntrace, 32) * a.uni_bs + (l - f * a.uni_bs);
  }
  __device__ __forceinline__ int bs(int t) const { return a.uni_nT ? a.uni_bs : __ldg(a.tpts + t) * a.nv; }
  __device__ __forceinline__ long long toff(int t) const {
    return a.uni_nT ? (long long)t * a.uni_bs : __ldg(a.toff + t);
  }
  __device__ __forceinline__ long long poff(int t) const {
    return a.uni_nT ? (long long)t * a.uni_bs * a.uni_bs : __ldg(a.poff + t);
  }
};

// FP32 to FP64 by the integer pipes (exact; zeros, subnormals, infinities and NaN by the conversion
// instruction, which shares the FP64 pipe)
__device__ __forceinline__ double any_widen(float x) {
  const unsigned u = __float_as_uint(x), e = (u >> 23) & 255u;
  if (e == 0u || e == 255u) return (double)x;
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))), (int)(u << 29));
}
__device__ __forceinline__ double any_widen(double x) { return x; }

// out[d] = base[d] - (or, without base, +) the sum of the element-view entries of trace value d, over
// [x0, x1); four values per thread in flight (their table entries, then the values themselves)
template <typename T>
__device__ void any_gather(const CycleArgs& a, const double* base, double* out, size_t x0, size_t x1) {
  const T* yv = reinterpret_cast<const T*>(a.yv);
  for (size_t xb = x0 + threadIdx.x; xb < x1; xb += 4 * PG_THREADS) {
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    if (a.uni_nT) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const size_t d = xb + (size_t)u * PG_THREADS;
        if (d >= x1) break;
        const int t = (int)(d / a.uni_bs), b = (int)(d % a.uni_bs);
#pragma unroll
        for (int sd = 0; sd < 2; ++sd) {
          const int e = __ldg(a.sides + 4 * t + 2 * sd), f = __ldg(a.sides + 4 * t + 2 * sd + 1);
          if (e >= 0)
            s[u] += any_widen(__ldcg(yv + (size_t)FR_IDX(e, a.Eim, 33) * a.uni_nT + FR_IDX(f, 4, 34) * a.uni_bs + b));
        }
      }
    } else {
      long long c[4], c1[4];
      int most = 0;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const size_t d = xb + (size_t)u * PG_THREADS;
        c[u] = d < x1 ? __ldg(a.vptr + d) : 0;
        c1[u] = d < x1 ? __ldg(a.vptr + d + 1) : 0;
        most = max(most, (int)(c1[u] - c[u]));
      }
      for (int i = 0; i < most; ++i) {
        long long ix[4];
        T v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) ix[u] = c[u] + i < c1[u] ? __ldg(a.vidx + c[u] + i) : -1;
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = ix[u] >= 0 ? __ldcg(yv + FR_IDX(ix[u], a.nview, 35)) : T(0);
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (ix[u] >= 0) s[u] += any_widen(v[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const size_t d = xb + (size_t)u * PG_THREADS;
      if (d < x1) out[d] = base ? __ldcg(base + d) - s[u] : s[u];
    }
  }
}

// y_k = S_k x_k over this warp's run of rows (X: T, the preconditioned vector, or double, x itself).
// The element's trace values are staged in the warp's shared memory, those of the next element
// loaded meanwhile; then 32 rows at a time, four lanes per row and four rows per lane, each lane
// every fourth 16-byte vector of its rows (scalar where the rows do not start on vectors).  Short
// FP64 rows go one per lane: their lane sums would cost the FP64 pipe more than the products.
template <typename T, typename X>
__device__ void any_matvec(const CycleArgs& a, const X* x, T* xs) {
  constexpr int VW = 16 / (int)sizeof(T), PF = 4;  // PF: values per lane of a next element loaded ahead
  struct alignas(16) Vec {
    T v[VW];
  };
  const AnyShape sh{a};
  const int lane = threadIdx.x & 31, r8 = lane >> 2, c4 = lane & 3;
  const long long W = (long long)gridDim.x * PG_WARPS, w = (long long)blockIdx.x * PG_WARPS + (threadIdx.x >> 5);
  const long long s0 = a.sumTT / W * w + a.sumTT % W * w / W, s1 = a.sumTT / W * (w + 1) + a.sumTT % W * (w + 1) / W;
  if (s0 >= s1) return;
  int lo = 0, hi = a.Eim - 1;  // the element that holds value s0
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (sh.offD(mid) <= s0) lo = mid;
    else hi = mid - 1;
  }
  const T* S = reinterpret_cast<const T*>(a.S);
  T* yv = reinterpret_cast<T*>(a.yv);
  auto value = [&](int k, long long o, int l) -> T {
    const long long g = sh.gmap(k, o, l);
    return g >= 0 ? T(__ldcg(x + g)) : T(0);
  };
  T nx[PF];
  bool have = false;  // nx holds the first 32 PF values of element k
  for (int k = lo; k < a.Eim; ++k) {
    const int nT = sh.nT(k);
    const long long od = sh.offD(k), o = sh.offs(k);
    if (od >= s1) break;
    // rows whose first value lies in [s0, s1)
    const int ra = od >= s0 ? 0 : (int)((s0 - od + nT - 1) / nT);
    const int rb = (int)min((long long)nT, (s1 - od + nT - 1) / nT);
    __syncwarp();
    if (ra < rb) {
#pragma unroll
      for (int q = 0; q < PF; ++q)
        if (lane + 32 * q < nT) xs[lane + 32 * q] = have ? nx[q] : value(k, o, lane + 32 * q);
      for (int l = lane + 32 * PF; l < nT; l += 32) xs[l] = value(k, o, l);
    }
    have = k + 1 < a.Eim && od + (long long)nT * nT < s1;
    if (have) {
      const int nT1 = sh.nT(k + 1);
      const long long o1 = sh.offs(k + 1);
#pragma unroll
      for (int q = 0; q < PF; ++q)
        if (lane + 32 * q < nT1) nx[q] = value(k + 1, o1, lane + 32 * q);
    }
    if (ra >= rb) continue;
    __syncwarp();
    const T* Sk = S + od;
    const bool vec = nT % VW == 0 && od % VW == 0;
    if (sizeof(T) == 8 && nT <= 16) {
      for (int r = ra + lane; r < rb; r += 32) {
        T acc = T(0);
        for (int c = 0; c < nT; ++c) acc = fma(__ldg(Sk + (size_t)r * nT + c), xs[c], acc);
        yv[o + r] = acc;
      }
      continue;
    }
    for (int r0 = ra; r0 < rb; r0 += 32) {
      T acc[4];
      const T* row[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        acc[u] = T(0);
        const int r = r0 + r8 + 8 * u;
        row[u] = Sk + (size_t)(r < rb ? r : rb - 1) * nT;  // a row past the end repeats the last one
      }
      if (vec) {
#pragma unroll 2
        for (int c = c4 * VW; c < nT; c += 4 * VW) {
          const Vec xv = *reinterpret_cast<const Vec*>(xs + c);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const PGVec<T, VW> sv = pg_ld_stream<T, VW>(row[u] + c);
#pragma unroll
            for (int q = 0; q < VW; ++q) acc[u] = fma(sv.v[q], xv.v[q], acc[u]);
          }
        }
      } else {
        for (int c = c4; c < nT; c += 4) {
          const T xv = xs[c];
#pragma unroll
          for (int u = 0; u < 4; ++u) acc[u] = fma(__ldg(row[u] + c), xv, acc[u]);
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], 1);
        acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], 2);
        const int r = r0 + r8 + 8 * u;
        if (c4 == 0 && r < rb) yv[o + r] = acc[u];
      }
    }
  }
}

// z = P^-1 v over the trace units [t0, t1), in the block precision.  Units of up to 8 values one per
// thread; up to 32 one per warp and lane a row, two units' rows in flight; larger ones one per warp
// with a lane on every 32nd row.  tid0, nthr: the threads that take part
template <typename T>
__device__ void any_precond(const CycleArgs& a, const double* v, T* z, int t0, int t1, int tid0, int nthr) {
  constexpr int VW = 16 / (int)sizeof(T);
  const AnyShape sh{a};
  const T* P = reinterpret_cast<const T*>(a.Pinv);
  if (a.bsmax <= 8) {
    for (int t = t0 + tid0; t < t1; t += nthr) {
      const int bs = sh.bs(t);
      const long long o = sh.toff(t);
      const T* Pt = P + sh.poff(t);
      T x[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) x[c] = c < bs ? T(v[o + c]) : T(0);
      for (int r = 0; r < bs; ++r) {
        T s = T(0);
#pragma unroll
        for (int c = 0; c < 8; ++c)
          if (c < bs) s = fma(__ldg(Pt + r * bs + c), x[c], s);
        z[o + r] = s;
      }
    }
    return;
  }
  const int lane = threadIdx.x & 31, nw = nthr >> 5;
  constexpr int RV = 24 / VW;  // vectors of a row held in registers
  if (sizeof(T) == 4 && a.bsmax <= 24) {
    for (int t = t0 + (tid0 >> 5); t < t1; t += 2 * nw) {
      PGVec<T, VW> row[2][RV];
      T x[2];
      int bs[2];
      long long o[2];
      bool ok[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int tt = t + h * nw < t1 ? t + h * nw : t;
        bs[h] = sh.bs(tt);
        o[h] = sh.toff(tt);
        const long long po = sh.poff(tt);
        ok[h] = bs[h] % VW == 0 && po % VW == 0;
        x[h] = lane < bs[h] ? T(v[o[h] + lane]) : T(0);
        const T* pr = P + po + (size_t)(lane < bs[h] ? lane : 0) * bs[h];
#pragma unroll
        for (int c = 0; c < RV; ++c) {
          if (ok[h] && c * VW < bs[h]) {
            row[h][c] = pg_ld_stream<T, VW>(pr + c * VW);
          } else {
#pragma unroll
            for (int e = 0; e < VW; ++e) row[h][c].v[e] = c * VW + e < bs[h] ? __ldg(pr + c * VW + e) : T(0);
          }
        }
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        T s = T(0);
#pragma unroll
        for (int c = 0; c < RV * VW; ++c)
          if (c < bs[h]) s = fma(row[h][c / VW].v[c % VW], __shfl_sync(0xffffffffu, x[h], c), s);
        if (lane < bs[h] && (h == 0 || t + nw < t1)) z[o[h] + lane] = s;
      }
    }
    return;
  }
  for (int t = t0 + (tid0 >> 5); t < t1; t += nw) {
    const int bs = sh.bs(t);
    const long long o = sh.toff(t), po = sh.poff(t);
    const bool vec = bs % VW == 0 && po % VW == 0;
    T x[4], acc[4];
    const T* row[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = lane + 32 * q;
      x[q] = i < bs ? T(v[o + i]) : T(0);
      acc[q] = T(0);
      row[q] = P + po + (size_t)(i < bs ? i : 0) * bs;
    }
#pragma unroll
    for (int qc = 0; qc < 4; ++qc) {
      const int cn = min(32, bs - 32 * qc);
      if (cn <= 0) break;
      if (vec) {
#pragma unroll 4
        for (int c = 0; c < cn; c += VW) {
          T xv[VW];
#pragma unroll
          for (int e = 0; e < VW; ++e) xv[e] = __shfl_sync(0xffffffffu, x[qc], c + e);
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (32 * q < bs) {
              const PGVec<T, VW> pv = pg_ld_stream<T, VW>(row[q] + 32 * qc + c);
#pragma unroll
              for (int e = 0; e < VW; ++e) acc[q] = fma(pv.v[e], xv[e], acc[q]);
            }
        }
      } else {
        for (int c = 0; c < cn; ++c) {
          const T xv = __shfl_sync(0xffffffffu, x[qc], c);
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (32 * q < bs) acc[q] = fma(__ldg(row[q] + 32 * qc + c), xv, acc[q]);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (lane + 32 * q < bs) z[o + lane + 32 * q] = acc[q];
  }
}

// x += sum_{i<k} y_i Z_i over [x0, x1) (FP64 sums of block-precision vectors)
template <typename T>
__device__ void any_update_x(const T* Z, size_t n, const double* y, int k, double* x, size_t x0, size_t x1) {
  for (size_t i = x0 + threadIdx.x; i < x1; i += PG_THREADS) {
    double s0 = 0.0, s1 = 0.0;
    int j = 0;
    for (; j + 8 <= k; j += 8) {
      T v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = Z[(size_t)(j + u) * n + i];
#pragma unroll
      for (int u = 0; u < 8; u += 2) {
        s0 = fma(y[j + u], any_widen(v[u]), s0);
        s1 = fma(y[j + u + 1], any_widen(v[u + 1]), s1);
      }
    }
    for (; j < k; ++j) s0 = fma(y[j], any_widen(Z[(size_t)j * n + i]), s0);
    x[i] += s0 + s1;
  }
}

constexpr int ANY_CLUSTER = 8;
template <typename T>
constexpr size_t any_smem() {
  return (sizeof(PGShared<double>) + 15) / 16 * 16 + (size_t)PG_WARPS * ANY_MAXT * sizeof(T);
}

// forms: a cooperative grid, where cancellation asks for the second Gram-Schmidt pass; one cluster of
// ANY_CLUSTER CTAs, and a grid for small systems, which make it always
enum { ANY_GRID = 0, ANY_ONE_CLUSTER = 1, ANY_GRID_SMALL = 2 };
template <typename T, int FORM>
__global__ void __launch_bounds__(PG_THREADS, 1) k_gmres_cycle_any(const __grid_constant__ CycleArgs a) {
  constexpr bool CLUSTER = FORM == ANY_ONE_CLUSTER, TEST = FORM == ANY_GRID;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PGShared<double>& sh = *reinterpret_cast<PGShared<double>*>(smem_raw);
  T* xs = reinterpret_cast<T*>(smem_raw + (sizeof(PGShared<double>) + 15) / 16 * 16) + (threadIdx.x >> 5) * ANY_MAXT;
  const AnyShape lay{a};
  const int tid = threadIdx.x;
  const size_t n = a.n;
  // trace units of this CTA: about n / gridDim.x values each
  auto first_unit = [&](int b) -> int {
    if (a.uni_nT) return (int)((long long)b * a.ntrace / gridDim.x);
    const long long want = (long long)b * (long long)n / gridDim.x;
    int lo = 0, hi = a.ntrace;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (__ldg(a.toff + mid) < want) lo = mid + 1;
      else hi = mid;
    }
    return lo;
  };
  const int t0 = first_unit(blockIdx.x), t1 = blockIdx.x + 1 == gridDim.x ? a.ntrace : first_unit(blockIdx.x + 1);
  const size_t x0 = (size_t)lay.toff(t0), x1 = t1 == a.ntrace ? n : (size_t)lay.toff(t1);
  unsigned epoch = 0;
  int par = 0;
  const size_t pstride = (size_t)PG_ND * gridDim.x;
  double *V = a.V, *partial = a.partial;
  T* Z = reinterpret_cast<T*>(a.Z);
  auto zrow = [&](int j) { return Z + (size_t)FR_IDX(j, GM_MAXM, 30) * n; };
  auto sync = [&]() -> bool {
    if constexpr (CLUSTER) {
      __syncthreads();
      asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
      return true;
    } else {
      return pg_sync(sh, a.bar, epoch);
    }
  };
  const int xz = a.dyn ? a.dyn[0] : a.x_zero;
  const int mm = a.dyn ? a.dyn[1] : a.m;
  // r0 = t - L x into V_0 (x = 0: r0 = t); beta = ||r0||, bnorm = ||t||
  if (!xz) {
    any_matvec<T, double>(a, a.x, xs);
    if (!sync()) return;
    any_gather<T>(a, a.t, V, x0, x1);
  } else {
    for (size_t x = x0 + tid; x < x1; x += PG_THREADS) V[x] = __ldcg(a.t + x);
  }
  __syncthreads();
  pg_block_sq(sh, V, a.t, x0, x1, partial + par * pstride);
  if (!sync()) return;
  pg_reduce(sh, 2, partial + par * pstride);
  par ^= 1;
  if (tid == 0) {
    const double beta = sqrt(sh.dot[0]);
    sh.beta = beta;
    sh.bnorm = sqrt(sh.dot[1]);
    sh.g[0] = beta;
    sh.res = beta;
    sh.hn = beta;
    sh.k = 0;
    sh.conv = 0;
    sh.nan = 0;
    sh.done = 0;
    sh.corr = 0;
    sh.invT = beta > 0.0 ? 1.0 / beta : 0.0;
    if (!(beta == beta)) {
      sh.nan = 1;
      sh.done = 1;
    } else if (beta <= a.rtol * sh.bnorm || beta == 0.0) {
      sh.conv = 1;
      sh.done = 1;
    }
  }
  __syncthreads();
  if (!sh.done) {
    for (int j = 0;; ++j) {
      double* vj = V + (size_t)j * n;
      double* w = V + (size_t)(j + 1) * n;
      // (A) lane 0 of warp 0: Givens rotation of column j-1; warps 1..: finish v_j, z_j = P^-1 v_j.
      // Pass mm only ends the cycle: v_mm and z_mm are not needed, and Z has GM_MAXM rows.
      if (j > 0 && tid == 0) pg_givens(sh, j - 1, a.rtol, mm);
      if (tid >= 32 && j < mm) {
        pg_finish(V, n, sh.cf, sh.corr ? j : 0, sh.invT, vj, x0, x1);
        pg_sync_workers();
        any_precond<T>(a, vj, zrow(j), t0, t1, tid - 32, PG_THREADS - 32);
      }
      if (!sync()) return;
      __syncthreads();
      if (sh.done) break;
      // (B) y_k = S_k z_k
      any_matvec<T, T>(a, zrow(j), xs);
      if (!sync()) return;
      // (C) w = L z, h = V^T w (and ||w||^2)
      any_gather<T>(a, nullptr, w, x0, x1);
      double* part = partial + par * pstride;
      pg_block_dots<double>(sh, V, n, j + (TEST ? 2 : 1), w, x0, x1, part);
      if (!sync()) return;
      pg_reduce(sh, j + (TEST ? 2 : 1), part);
      par ^= 1;
      if constexpr (!TEST) {
        for (int i = tid; i <= j; i += PG_THREADS) {
          sh.hc[i] = sh.dot[i];
          sh.cf[i] = sh.dot[i];
        }
      } else if (tid < 32) {
        double hh = 0.0;
        for (int i = tid; i <= j; i += 32) {
          const double h = sh.dot[i];
          hh += h * h;
          sh.hc[i] = h;
          sh.cf[i] = h;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
          if (o <= j) hh += __shfl_xor_sync(0xffffffffu, hh, o);  // lanes above j hold zeros
        if (tid == 0) {
          const double n0 = sh.dot[j + 1];
          const int corr = hh <= 0.5 * n0 ? 1 : 0;
          sh.corr = corr;
          if (corr) {
            const double hn = sqrt(n0 - hh);
            sh.hc[j + 1] = hn;
            sh.invT = hn != 0.0 ? 1.0 / hn : 0.0;
          }
        }
      }
      __syncthreads();
      // little cancellation (the test of the short kernels): one pass, w' formed with v_{j+1}
      if (TEST && sh.corr) continue;
      // (D) w' = w - V h, then d = V^T w' and ||w'||^2
      pg_subtract(V, n, sh.cf, j, w, x0, x1);
      part = partial + par * pstride;
      pg_block_dots<double>(sh, V, n, j + 2, w, x0, x1, part);
      if (!sync()) return;
      pg_reduce(sh, j + 2, part);
      par ^= 1;
      if (tid < 32) {
        double dd = 0.0;
        for (int i = tid; i <= j; i += 32) {
          const double d = sh.dot[i];
          dd += d * d;
          sh.hc[i] += d;
          sh.cf[i] = d;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) dd += __shfl_xor_sync(0xffffffffu, dd, o);
        if (tid == 0) {
          const double n1 = sh.dot[j + 1];
          sh.corr = dd <= 0.25 * n1 ? 1 : 0;
          if (sh.corr) sh.hc[j + 1] = sqrt(n1 - dd);
        }
      }
      __syncthreads();
      if (!sh.corr) {  // severe cancellation: form w'' = w' - V d now and sum its norm
        pg_subtract(V, n, sh.cf, j, w, x0, x1);
        part = partial + par * pstride;
        pg_block_sq(sh, w, (const double*)nullptr, x0, x1, part);
        if (!sync()) return;
        pg_reduce(sh, 1, part);
        par ^= 1;
        if (tid == 0) sh.hc[j + 1] = sqrt(sh.dot[0]);
      }
      if (tid == 0) sh.invT = sh.hc[j + 1] != 0.0 ? 1.0 / sh.hc[j + 1] : 0.0;
      __syncthreads();
    }
  }
  // y = H^{-1} g, x += Z y
  const int k = sh.k;
  if (tid == 0) {
    for (int i = k - 1; i >= 0; --i) {
      double s = sh.g[i];
      for (int c = i + 1; c < k; ++c) s -= sh.H[i * GM_MAXM + c] * sh.y[c];
      sh.y[i] = s * sh.rdi[i];
    }
  }
  __syncthreads();
  if (k > 0) any_update_x<T>(Z, n, sh.y, k, a.x, x0, x1);
  if (a.true_res) {  // ||t - L x|| (V_0 as scratch)
    if (!sync()) return;
    any_matvec<T, double>(a, a.x, xs);
    if (!sync()) return;
    any_gather<T>(a, a.t, V, x0, x1);
    __syncthreads();
    pg_block_sq(sh, V, (const double*)nullptr, x0, x1, partial + par * pstride);
    if (!sync()) return;
    pg_reduce(sh, 1, partial + par * pstride);
  }
  if (blockIdx.x == 0 && tid == 0) {
    GmresState* st = a.st;
    st->beta = a.true_res ? sqrt(sh.dot[0]) : sh.res;
    st->bnorm = sh.bnorm;
    st->res = sh.res;
    st->hn = sh.hn;
    st->k = k;
    st->kdone = k;
    st->converged = sh.conv;
    st->nan = sh.nan;
  }
}

template <typename T, int NT, int BS, bool SB>
cudaError_t launch_cycle(const FusedArgs& a, int grid, cudaStream_t s) {
  const size_t smem = sizeof(PGShared<T>);
  cudaError_t e = cudaFuncSetAttribute(k_gmres_cycle<T, NT, BS, SB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  void* args[] = {const_cast<FusedArgs*>(&a)};
  (hfr::count_launch(),
   e = cudaLaunchCooperativeKernel((const void*)k_gmres_cycle<T, NT, BS, SB>, dim3(grid), dim3(PG_THREADS), args, smem, s));
  return e;
}

template <typename T, int NT, int BS, bool SB>
int occupancy_of() {
  int nb = 0;
  const size_t smem = sizeof(PGShared<T>);
  if (cudaFuncSetAttribute(k_gmres_cycle<T, NT, BS, SB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
      cudaSuccess)
    return 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_gmres_cycle<T, NT, BS, SB>, PG_THREADS, smem) != cudaSuccess)
    return 0;
  return nb;
}

typedef cudaError_t (*CycleFn)(const FusedArgs&, int, cudaStream_t);

// s_bf16: the trace operator S is stored in BF16 (FP32 blocks, basis and arithmetic otherwise)
CycleFn pick(int prec_bytes, int nT, int bs, int* occ, bool s_bf16 = false) {
#define HFR_PG(T_, NT_, BS_, SB_)                  \
  if (nT == NT_ && bs == BS_) {                    \
    *occ = occupancy_of<T_, NT_, BS_, SB_>();      \
    return launch_cycle<T_, NT_, BS_, SB_>;        \
  }
  if (prec_bytes == 4 && s_bf16) {
    HFR_PG(float, 64, 16, true)
    HFR_PG(float, 80, 20, true)
    HFR_PG(float, 48, 12, true)
  } else if (prec_bytes == 4) {
    HFR_PG(float, 64, 16, false)
    HFR_PG(float, 80, 20, false)
    HFR_PG(float, 48, 12, false)
  } else {
    HFR_PG(double, 64, 16, false)
    HFR_PG(double, 80, 20, false)
    HFR_PG(double, 48, 12, false)
  }
#undef HFR_PG
  *occ = 0;
  return nullptr;
}

}  // namespace

size_t fused_partial_doubles(int max_blocks) { return (size_t)2 * PG_ND * (size_t)max_blocks; }  // >= T slots

int fused_gmres_grid(int prec_bytes, int nT, int bs) {
  int dev = 0, coop = 0, nsm = 0, occ = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) return 0;
  if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  if (!pick(prec_bytes, nT, bs, &occ) || occ < 1) return 0;
  return nsm;  // one CTA per SM
}

int run_gmres_fused(const FusedArgs& base, int prec_bytes, int grid, double rtol, int restart, int maxit,
                    GmresResult* res, int* timed_out, cudaStream_t s, const int* dev_status, int* host_status) {
  int occ = 0;
  const int bs = (int)(base.n / (size_t)base.ntrace);
  CycleFn fn = pick(prec_bytes, base.nT, bs, &occ, base.s_bf16 != 0);
  *timed_out = 0;
  if (!fn || grid < 1) return -1;
  const int m = restart > GM_MAXM ? GM_MAXM : (restart < 1 ? 1 : restart);
  FusedArgs a = base;
  a.rtol = rtol;
  if (cudaMemsetAsync(a.x, 0, a.n * sizeof(double), s) != cudaSuccess) return -1;
  int total = 0;
  bool first = true, first_cycle = true;
  for (;;) {
    a.m = m < maxit - total ? m : maxit - total;
    a.x_zero = first ? 1 : 0;
    first = false;
    if (cudaMemsetAsync(a.bar, 0, 2 * sizeof(unsigned), s) != cudaSuccess) return -1;
    if (fn(a, grid, s) != cudaSuccess) return -1;
    GmresHead hs;
    unsigned flags[2] = {0u, 0u};
    if (cudaMemcpyAsync(&hs, a.st, sizeof(GmresHead), cudaMemcpyDeviceToHost, s) != cudaSuccess) return -1;
    if (cudaMemcpyAsync(flags, a.bar, sizeof(flags), cudaMemcpyDeviceToHost, s) != cudaSuccess) return -1;
    if (dev_status && first_cycle &&
        cudaMemcpyAsync(host_status, dev_status, 2 * sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess)
      return -1;
    first_cycle = false;
    if (cudaStreamSynchronize(s) != cudaSuccess) return -1;
    if (flags[1] != 0u) {
      *timed_out = 1;
      res->iterations = total;
      res->converged = 0;
      res->nan = 0;
      return 0;
    }
    total += hs.k;
    res->bnorm = hs.bnorm;
    res->rel = hs.bnorm > 0.0 ? hs.beta / hs.bnorm : 0.0;
    res->iterations = total;
    res->nan = hs.nan;
    res->converged = hs.converged;
    if (hs.nan || hs.converged || total >= maxit || hs.k == 0) return 0;
  }
}

cudaError_t launch_gmres_cycle(const FusedArgs& a, int prec_bytes, int grid, cudaStream_t s) {
  int occ = 0;
  const int bs = (int)(a.n / (size_t)(a.ntrace > 0 ? a.ntrace : 1));
  CycleFn fn = pick(prec_bytes, a.nT, bs, &occ, a.s_bf16 != 0);
  if (!fn || grid < 1) return cudaErrorInvalidValue;
  return fn(a, grid, s);
}

template <typename T, int FORM>
static cudaError_t any_config(int grid, cudaStream_t s, cudaLaunchConfig_t& cfg, cudaLaunchAttribute (&at)[1]) {
  cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(PG_THREADS);
  cfg.dynamicSmemBytes = any_smem<T>();
  cfg.stream = s;
  if (FORM == ANY_ONE_CLUSTER) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = ANY_CLUSTER;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
  } else {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
  }
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaFuncSetAttribute(k_gmres_cycle_any<T, FORM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)any_smem<T>());
}

template <typename T, int FORM>
static cudaError_t launch_any(const CycleArgs& a, const CyclePlan& p, cudaStream_t s) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[1];
  const cudaError_t e = any_config<T, FORM>(p.grid, s, cfg, at);
  if (e != cudaSuccess) return e;
  hfr::count_launch();
  return cudaLaunchKernelEx(&cfg, k_gmres_cycle_any<T, FORM>, a);
}
template <typename T>
static cudaError_t launch_form(const CycleArgs& a, const CyclePlan& p, cudaStream_t s) {
  if (p.form == ANY_ONE_CLUSTER) return launch_any<T, ANY_ONE_CLUSTER>(a, p, s);
  if (p.form == ANY_GRID_SMALL) return launch_any<T, ANY_GRID_SMALL>(a, p, s);
  return launch_any<T, ANY_GRID>(a, p, s);
}

// one cluster of the cycle can be resident on the device
template <typename T>
static bool cluster_fits() {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[1];
  int n = 0;
  return any_config<T, ANY_ONE_CLUSTER>(ANY_CLUSTER, nullptr, cfg, at) == cudaSuccess &&
         cudaOccupancyMaxActiveClusters(&n, k_gmres_cycle_any<T, ANY_ONE_CLUSTER>, &cfg) == cudaSuccess && n >= 1;
}

cudaError_t launch_cycle_any(const CycleArgs& a, int prec_bytes, const CyclePlan& p, cudaStream_t s) {
  if (p.grid < 1) return cudaErrorInvalidValue;
  return prec_bytes == 4 ? launch_form<float>(a, p, s) : launch_form<double>(a, p, s);
}

// The cluster form for small systems, by the multiply-adds of an iteration (S once, the FP64 vectors some
// forty times): above the line, eight SMs take longer for them than the grid barriers of the whole
// device cost (four per iteration), sooner in FP64, whose pipe is the narrow one.  Time per iteration of
// a cycle of 20, cluster / grid / short kernels, in us:
//   FP32  25 000: 26.6 / 29.6 / 63   98 000: 29.3 / 30.5 / 65   154 000: 35.9 / 31.0 / 66   229 000: 48 / 31 / 66
//   FP64  25 000: 28.0 / 30.2 / 67   37 000: 28.6 / 30.4 / 68   90 000: 35.4 / 31.8 / 67   187 000: 52 / 43 / 109
// (scalar elements of 8 x 8 to 32 x 32, p = 1 to 3; the last of FP64: wall elements).  The lines are where
// the scalar elements cross; shapes of several variables in FP64 cross below it (EDAC, p = 2, 18 000: 36.7 / 32.5
// / 70) and FP32 faces of two values sooner (p = 1, 90 000: 33.5 / 30.7 / 64).
CyclePlan cycle_plan(int prec_bytes, const CycleArgs& a) {
  CyclePlan p;
  int dev = 0, coop = 0, nsm = 0, occ = 0;
  // what the kernel holds of an element (a warp's shared memory) and of a trace unit (registers)
  if (a.ntrace <= 0 || a.Eim <= 0 || a.bsmax > 128 || a.nTmax > ANY_MAXT) return p;
  // Large uniform systems of FP64 blocks with faces of more than 16 values (Navier-Stokes, p = 5): the
  // short kernels' uniform mat-vec and preconditioner spend fewer FP64 instructions on lane sums and
  // idle lanes, which outweighs the launches above some 10^8 values of S.  Time per iteration, single
  // launch against short kernels: 96 x 96 elements (0.85 10^8) 416 / 448 us, 128 x 128 (1.5 10^8)
  // 703 / 679 us, where the second Gram-Schmidt pass is not needed 380 / 385 and 637 / 586 us.
  if (prec_bytes == 8 && a.uni_nT > 0 && a.uni_bs > 16 && a.sumTT > 100000000LL) return p;
  if (cudaGetDevice(&dev) != cudaSuccess) return p;
  if (a.sumTT + 40 * (long long)a.n <= (prec_bytes == 4 ? 100000 : 40000)) {
    const bool ok = prec_bytes == 4 ? cluster_fits<float>() : cluster_fits<double>();
    if (ok) {
      p.grid = ANY_CLUSTER;
      p.form = ANY_ONE_CLUSTER;
      return p;
    }
    cudaGetLastError();
  }
  if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) return p;
  if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return p;
  auto fits = [&](auto kern, size_t smem) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess &&
           cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, PG_THREADS, smem) == cudaSuccess && occ >= 1;
  };
  // The test for the second Gram-Schmidt pass sits on the chain of every iteration (0.5 us).  Systems of
  // fewer than some 25 000 trace values make the pass always: where the test never lets them off they
  // lose up to 1.3 % by it, where it does the single launch is ahead of the short kernels by 40 % either way.
  // Per iteration with the test / without, in us, ten times the explicit step and 300 times: EFR p = 4,
  // 15 000 values 47.9 / 47.5 and 40.0 / 47.3, 64 500 values 59.9 / 60.5 and 49.0 / 60.4, 459 000 values
  // 244.7 / 244.9 and 220.2 / 245.9 (short kernels 236.3); scalar, p = 2, FP64, 14 000 values 35.7 / 35.4; one
  // cluster, 64 scalar elements 27.8 / 26.5.
  const bool small = a.n < 25000;
  const bool ok = prec_bytes == 4 ? (small ? fits(k_gmres_cycle_any<float, ANY_GRID_SMALL>, any_smem<float>())
                                           : fits(k_gmres_cycle_any<float, ANY_GRID>, any_smem<float>()))
                                  : (small ? fits(k_gmres_cycle_any<double, ANY_GRID_SMALL>, any_smem<double>())
                                           : fits(k_gmres_cycle_any<double, ANY_GRID>, any_smem<double>()));
  if (ok) {
    p.grid = nsm;  // one CTA per SM
    p.form = small ? ANY_GRID_SMALL : ANY_GRID;
  }
  return p;
}

int run_gmres_any(const CycleArgs& base, int prec_bytes, const CyclePlan& p, double rtol, int restart, int maxit,
                  bool true_res, GmresResult* res, int* timed_out, cudaStream_t s) {
  const int m = restart > GM_MAXM ? GM_MAXM : (restart < 1 ? 1 : restart);
  CycleArgs a = base;
  a.rtol = rtol;
  a.true_res = true_res ? 1 : 0;
  *timed_out = 0;
  if (cudaMemsetAsync(a.x, 0, a.n * sizeof(double), s) != cudaSuccess) return -1;
  int total = 0;
  for (bool first = true;; first = false) {
    a.m = m < maxit - total ? m : maxit - total;
    a.x_zero = first ? 1 : 0;
    if (total + a.m >= maxit) a.true_res = 1;  // the cycle that may end at the limit: its residual is reported
    if (cudaMemsetAsync(a.bar, 0, 2 * sizeof(unsigned), s) != cudaSuccess) return -1;
    if (launch_cycle_any(a, prec_bytes, p, s) != cudaSuccess) return -1;
    GmresHead hs;
    unsigned flags[2] = {0u, 0u};
    if (cudaMemcpyAsync(&hs, a.st, sizeof(GmresHead), cudaMemcpyDeviceToHost, s) != cudaSuccess) return -1;
    if (cudaMemcpyAsync(flags, a.bar, sizeof(flags), cudaMemcpyDeviceToHost, s) != cudaSuccess) return -1;
    if (cudaStreamSynchronize(s) != cudaSuccess) return -1;
    res->iterations = total;
    res->nan = res->converged = 0;
    if (flags[1] != 0u) {
      *timed_out = 1;
      return 0;
    }
    total += hs.k;
    res->bnorm = hs.bnorm;
    res->rel = hs.bnorm > 0.0 ? hs.beta / hs.bnorm : 0.0;
    res->iterations = total;
    res->nan = hs.nan;
    res->converged = hs.converged;
    if (hs.nan || hs.converged || total >= maxit || hs.k == 0) return 0;
  }
}

// ------------------------------------------------------------ inside a captured graph
__global__ void k_ga_begin(GmresGraphDev* d, int m, int maxit, cudaGraphConditionalHandle hw) {
  d->total = 0;
  d->cycles = 0;
  d->nan = 0;
  d->converged = 0;
  d->timeout = 0;
  d->dyn[0] = 1;
  d->dyn[1] = m < maxit ? m : maxit;
  cudaGraphSetConditional(hw, 1u);
}
__global__ void k_ga_after(GmresGraphDev* d, const GmresState* st, const unsigned* bar, int m, int maxit,
                           cudaGraphConditionalHandle hw) {
  int cont = 0;
  d->cycles += 1;
  if (bar[1] != 0u) {
    d->timeout = 1;
  } else {
    d->total += st->k;
    if (st->nan) d->nan = 1;
    d->converged = st->converged;
    cont = (st->nan || st->converged || d->total >= maxit || st->k == 0) ? 0 : 1;
    const int rem = maxit - d->total;
    d->dyn[0] = 0;
    d->dyn[1] = m < rem ? m : rem;
  }
  cudaGraphSetConditional(hw, (unsigned)cont);
}

cudaError_t capture_gmres_any(CycleArgs a, int prec_bytes, const CyclePlan& p, double rtol, int restart, int maxit,
                              GmresGraphDev* dev, cudaStream_t s, cudaStream_t sc, GmresGraphLaunches* counts) {
  const int m = restart > GM_MAXM ? GM_MAXM : (restart < 1 ? 1 : restart);
  a.rtol = rtol;
  a.m = m;
  a.x_zero = 1;
  a.true_res = 0;
  a.dyn = dev->dyn;
  cudaError_t e;
  const unsigned long long l0 = hfr::launch_count();
  cudaGraphConditionalHandle hw;
  if ((e = graph_conditional_handle(s, 0u, 0u, &hw)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(a.x, 0, a.n * sizeof(double), s)) != cudaSuccess) return e;
  (hfr::count_launch(), k_ga_begin<<<1, 1, 0, s>>>(dev, m, maxit, hw));
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  cudaGraph_t body = nullptr;
  if ((e = graph_add_conditional(s, hw, cudaGraphCondTypeWhile, &body)) != cudaSuccess) return e;
  const unsigned long long l1 = hfr::launch_count();
  if ((e = cudaStreamBeginCaptureToGraph(sc, body, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed)) != cudaSuccess)
    return e;
  e = cudaMemsetAsync(a.bar, 0, 2 * sizeof(unsigned), sc);
  if (e == cudaSuccess) e = launch_cycle_any(a, prec_bytes, p, sc);
  if (e == cudaSuccess) {
    (hfr::count_launch(), k_ga_after<<<1, 1, 0, sc>>>(dev, a.st, a.bar, m, maxit, hw));
    e = cudaGetLastError();
  }
  cudaGraph_t tmp = nullptr;
  const cudaError_t e2 = cudaStreamEndCapture(sc, &tmp);
  if (counts) {
    counts->fixed = (int)(l1 - l0);
    counts->cycle = (int)(hfr::launch_count() - l1);
    counts->residual = 0;
  }
  return e != cudaSuccess ? e : e2;
}

// Host side of the barrier self-test (declared in hfr_krylov.h).
int barrier_selftest(int nblocks, int absent, int rounds, double timeout_s, int* passed, int* timed_out,
                     cudaStream_t s) {
  *passed = 0;
  *timed_out = 0;
  int dev = 0, nsm = 0, per_sm = 0, coop = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return -1;
  if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return -1;
  if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess) return -1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_barrier_probe, 128, 0) != cudaSuccess) return -1;
  if (!coop || nblocks < 1 || nblocks > nsm * per_sm || rounds < 0) return -2;
  unsigned* bar = nullptr;
  int* dpass = nullptr;
  if (cudaMalloc((void**)&bar, 2 * sizeof(unsigned) + sizeof(int)) != cudaSuccess) return -1;
  dpass = reinterpret_cast<int*>(bar + 2);
  int rc = 0;
  unsigned flags[2] = {0u, 0u};
  unsigned long long tns = (unsigned long long)(timeout_s * 1e9);
  void* args[] = {&bar, &absent, &rounds, &tns, &dpass};
  if (cudaMemsetAsync(bar, 0, 2 * sizeof(unsigned) + sizeof(int), s) != cudaSuccess ||
      cudaLaunchCooperativeKernel((const void*)k_barrier_probe, dim3(nblocks), dim3(128), args, 0, s) != cudaSuccess ||
      cudaMemcpyAsync(flags, bar, sizeof(flags), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaMemcpyAsync(passed, dpass, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    rc = -1;
  cudaStreamSynchronize(s);
  cudaFree(bar);
  *timed_out = flags[1] != 0u;
  return rc;
}

}  // namespace hfr

#include "hfr_checked_unit.inc"
