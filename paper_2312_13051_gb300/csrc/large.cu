// Occupied states for large n (supercells, many-band models): Bloch Hamiltonian,
// Householder tridiagonalisation, bisection, inverse iteration, back-transform,
// and for the mixed path an FP64 Newton correction of the occupied block
// (Sec. I "exact diagonalization" at many k-points; Eq. 1 occupied bands).
//
// Each stage is its own kernel over a wave of W k-points, one CTA (or one thread
// per eigenpair) per k-point, with the wave's scratch in the context arena:
//   A[kw]   n x n complex, reduced in place; the unit Householder vectors u_c are
//           kept below the subdiagonal (column c, rows c+1..n-1)
//   dg, od  diagonal and |off-diagonal| of the real tridiagonal T' = D^dag T D
//   Dp      the unit phases D (x = Q D z maps eigenvectors z of T' to those of H)
//   lam, Z  eigenvalues (ascending) and eigenvectors of T' (Z[kw][row][col])
// T is the working precision of the reduction (double: FP64 path, float: mixed).
#include <float.h>

#include <algorithm>
#include <type_traits>

#include "ctagemm.cuh"
#include "df32.cuh"
#include "jacobi.cuh"
#include "launch.h"

namespace bw {

template <typename T>
__device__ __forceinline__ T lg_eps();
template <>
__device__ __forceinline__ double lg_eps<double>() { return 2.220446049250313e-16; }
template <>
__device__ __forceinline__ float lg_eps<float>() { return 1.1920929e-7f; }

// Warp-wide sum of a complex value.
template <typename T>
__device__ __forceinline__ cx<T> warp_csum(cx<T> v) {
  for (int o = 16; o > 0; o >>= 1) {
    v.re += __shfl_xor_sync(0xffffffffu, v.re, o);
    v.im += __shfl_xor_sync(0xffffffffu, v.im, o);
  }
  return v;
}


__device__ __forceinline__ void lg_kpoint(const LargeArgs& a, long long k, double f[3]) {
  if (a.f) {
    f[0] = a.f[3 * k]; f[1] = a.f[3 * k + 1]; f[2] = a.f[3 * k + 2];
  } else {
    const int i = int(k / a.plane.N), j = int(k - (long long)i * a.plane.N);
    plane_f(a.plane, i, j, f);
  }
}

__device__ __forceinline__ void split64(z64 x, c32& hi, c32& lo) {
  hi = c32(float(x.re), float(x.im));
  lo = c32(float(x.re - double(hi.re)), float(x.im - double(hi.im)));
}

// ---------------------------------------------------------------------------
// Stage 1: Bloch Hamiltonian of the wave's k-points (full Hermitian matrix).
// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_lg_build(LargeArgs a) {
  __shared__ __align__(16) unsigned char phs_raw[PHASE_CACHE * sizeof(z64)];
  z64* phs = reinterpret_cast<z64*>(phs_raw);
  const DevModel& md = a.model;
  const int n = a.n, tid = threadIdx.x, nt = blockDim.x;
  const int nRs = min(md.n_R, PHASE_CACHE);
  for (long long kw = blockIdx.x; kw < a.W; kw += gridDim.x) {
    if (std::is_same<T, double>::value && a.need && !a.need[kw]) continue;
    if (a.Hin) {  // explicit matrix: lower triangle mirrored, FP64 entries kept for the refinement
      const z64* Hm = a.Hin + a.h_off[a.idx[a.k0 + kw]];
      cx<T>* A = reinterpret_cast<cx<T>*>(a.A) + kw * (long long)n * n;
      c32* He = a.Hent ? reinterpret_cast<c32*>(a.Hent + kw * (long long)n * n) : nullptr;
      for (int r = tid >> 5; r < n; r += nt >> 5)
        for (int q = tid & 31; q <= r; q += 32) {
          z64 h = Hm[(long long)r * n + q];
          if (q == r) h.im = 0.0;
          A[(long long)r * n + q] = ccast<T>(h);
          A[(long long)q * n + r] = ccast<T>(conj(h));
          if (He) {
            c32 hi, lo;
            split64(h, hi, lo);
            He[2 * ((long long)r * n + q)] = hi;
            He[2 * ((long long)r * n + q) + 1] = lo;
            split64(conj(h), hi, lo);
            He[2 * ((long long)q * n + r)] = hi;
            He[2 * ((long long)q * n + r) + 1] = lo;
          }
        }
      __syncthreads();
      continue;
    }
    const long long k = a.k0 + kw * (a.kstride > 0 ? a.kstride : 1);
    double f[3];
    lg_kpoint(a, k, f);
    cx<T>* A = reinterpret_cast<cx<T>*>(a.A) + kw * (long long)n * n;
    for (long long e = tid; e < (long long)n * n; e += nt) A[e] = cx<T>(T(0), T(0));
    if (a.Hent && md.hop_tdf && !a.polish) {
      // mixed path: entries in double-float on the FP32 pipe (FP64-grade for the
      // refinement's residual, the FP32 matrix is the high part)
      cdf* phd = reinterpret_cast<cdf*>(phs);
      for (int r = tid; r < nRs; r += nt) phd[r] = cdf_from(bloch_phase(f, md.Rv + 3 * r));
      __syncthreads();
      for (int e = tid; e < md.n_ent; e += nt) {
        cdf acc(df(0.f), df(0.f));
        for (int h = md.ent_start[e]; h < md.ent_start[e + 1]; ++h) {
          const int r = md.hop_r[h];
          // one 16-byte load: the entries of neighbouring threads lie n_R hoppings apart, so
          // every load instruction touches a line per lane
          const float4 t4 = reinterpret_cast<const float4*>(md.hop_tdf)[h];
          cfma(acc, cdf(df(t4.x, t4.y), df(t4.z, t4.w)),
               r < nRs ? phd[r] : cdf_from(bloch_phase(f, md.Rv + 3 * r)));
        }
        A[(long long)md.ent_row[e] * n + md.ent_col[e]] = cx<T>(T(acc.re.hi), T(acc.im.hi));
        c32* dst = reinterpret_cast<c32*>(a.Hent + kw * (long long)md.n_ent + e);
        dst[0] = c32(acc.re.hi, acc.im.hi);
        dst[1] = c32(acc.re.lo, acc.im.lo);
      }
      __syncthreads();
      continue;
    }
    for (int r = tid; r < nRs; r += nt) phs[r] = bloch_phase(f, md.Rv + 3 * r);
    __syncthreads();
    for (int e = tid; e < md.n_ent; e += nt) {
      z64 acc(0.0, 0.0);
      for (int h = md.ent_start[e]; h < md.ent_start[e + 1]; ++h) {
        const int r = md.hop_r[h];
        const double2 t = reinterpret_cast<const double2*>(md.hop_t)[h];
        cfma(acc, z64(t.x, t.y), r < nRs ? phs[r] : bloch_phase(f, md.Rv + 3 * r));
      }
      if (a.polish) acc = a.scale * acc;
      A[(long long)md.ent_row[e] * n + md.ent_col[e]] = ccast<T>(acc);
      if (a.Hent) {  // FP64 entry as an unevaluated sum of two floats (hi, lo)
        c32 hi, lo;
        split64(acc, hi, lo);
        c32* dst = reinterpret_cast<c32*>(a.Hent + kw * (long long)md.n_ent + e);
        dst[0] = hi;
        dst[1] = lo;
        if (a.polish) a.H64[kw * (long long)md.n_ent + e] = acc;
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Stage 2: Householder reduction to tridiagonal form, one CTA per k-point.
// For column c, x = A[c+1:, c]; P = I - 2 u u^dagger with u ~ x - alpha e_1,
// alpha = -e^{i arg x_0} |x|, maps x to alpha e_1.  With p = A22 u, K = u^dag p
// and w = p - K u, the trailing block becomes A22 - 2 (u w^dag + w u^dag).
// The complex subdiagonal alpha_c is made real by D: D_0 = 1,
// D_{c+1} = D_c alpha_c / |alpha_c|, off-diagonal |alpha_c|.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_lg_tridiag(LargeArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int n = a.n, tid = threadIdx.x, nt = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nwarp = nt >> 5;
  cx<T>* u = reinterpret_cast<cx<T>*>(smem);          // n
  cx<T>* w = u + n;                                   // n
  cx<T>* al = w + n;                                  // n   complex subdiagonal
  double* red = reinterpret_cast<double*>(al + n);    // 64
  __shared__ double s_nrm2, s_x0re, s_x0im;
  __shared__ int s_skip;
  for (long long kw = blockIdx.x; kw < a.W; kw += gridDim.x) {
    if (std::is_same<T, double>::value && a.need && !a.need[kw]) continue;
    cx<T>* A = reinterpret_cast<cx<T>*>(a.A) + kw * (long long)n * n;
    T* dg = reinterpret_cast<T*>(a.dg) + kw * n;
    T* od = reinterpret_cast<T*>(a.od) + kw * n;
    cx<T>* Dp = reinterpret_cast<cx<T>*>(a.Dp) + kw * n;
    for (int c = 0; c + 2 < n; ++c) {
      const int m = n - c - 1;  // length of x
      double s = 0.0;
      for (int r = tid; r < m; r += nt) {
        const cx<T> x = A[(long long)(c + 1 + r) * n + c];
        u[r] = x;
        s += double(abs2(x));
      }
      s = block_sum(s, red);
      if (tid == 0) {
        s_nrm2 = s;
        s_x0re = double(u[0].re);
        s_x0im = double(u[0].im);
        s_skip = !(s - (s_x0re * s_x0re + s_x0im * s_x0im) > 0.0);
      }
      __syncthreads();
      const double nx = sqrt(s_nrm2), ax0 = hypot(s_x0re, s_x0im);
      if (s_skip) {  // already tridiagonal in this column: no reflection
        for (int r = tid; r < m; r += nt) A[(long long)(c + 1 + r) * n + c] = cx<T>(T(0), T(0));
        if (tid == 0) {
          al[c] = cx<T>(T(s_x0re), T(s_x0im));
          dg[c] = A[(long long)c * n + c].re;
        }
        __syncthreads();
        continue;
      }
      const double phr = ax0 > 0.0 ? s_x0re / ax0 : 1.0, phi = ax0 > 0.0 ? s_x0im / ax0 : 0.0;
      // v = x - alpha e1 with alpha = -ph |x|: v_0 = ph (|x0| + |x|); |v|^2 = (|x0|+|x|)^2 + tail
      const double tail = s_nrm2 - ax0 * ax0;
      const double v0m = ax0 + nx;
      const T inv = T(1.0 / sqrt(v0m * v0m + tail));
      __syncthreads();
      for (int r = tid; r < m; r += nt) {
        cx<T> v = u[r];
        if (r == 0) v = cx<T>(T(phr * v0m), T(phi * v0m));
        u[r] = inv * v;
      }
      __syncthreads();
      // p = A22 u: one warp per row, lanes along the row
      for (int r = warp; r < m; r += nwarp) {
        const cx<T>* row = A + (long long)(c + 1 + r) * n + (c + 1);
        cx<T> acc(T(0), T(0));
        for (int q = lane; q < m; q += 32) cfma(acc, row[q], u[q]);
        acc = warp_csum(acc);
        if (lane == 0) w[r] = acc;
      }
      __syncthreads();
      double kr = 0.0;
      for (int r = tid; r < m; r += nt) kr += double(u[r].re * w[r].re + u[r].im * w[r].im);
      kr = block_sum(kr, red);
      for (int r = tid; r < m; r += nt) w[r] = w[r] - T(kr) * u[r];
      __syncthreads();
      // A22 <- A22 - 2 (u w^dag + w u^dag)
      for (int r = warp; r < m; r += nwarp) {
        cx<T>* row = A + (long long)(c + 1 + r) * n + (c + 1);
        const cx<T> ur = u[r], wr = w[r];
        for (int q = lane; q < m; q += 32) row[q] = row[q] - T(2) * (ur * conj(w[q]) + wr * conj(u[q]));
      }
      if (tid == 0) {
        al[c] = cx<T>(T(-phr * nx), T(-phi * nx));
        dg[c] = A[(long long)c * n + c].re;
      }
      // keep u below the subdiagonal for the back-transform
      for (int r = tid; r < m; r += nt) A[(long long)(c + 1 + r) * n + c] = u[r];
      __syncthreads();
    }
    if (tid == 0) {
      if (n >= 2) {
        dg[n - 2] = A[(long long)(n - 2) * n + (n - 2)].re;
        al[n - 2] = A[(long long)(n - 1) * n + (n - 2)];
      }
      dg[n - 1] = A[(long long)(n - 1) * n + (n - 1)].re;
      // the last subdiagonal entry is not a reflector: clear it for the back-transform
      if (n >= 2) A[(long long)(n - 1) * n + (n - 2)] = cx<T>(T(0), T(0));
    }
    __syncthreads();
    // unit phases of the subdiagonal, then their prefix products (serial: cheap)
    for (int c = tid; c + 1 < n; c += nt) {
      const T aa = sqrt(abs2(al[c]));
      od[c] = aa;
      al[c] = aa > T(0) ? cx<T>(al[c].re / aa, al[c].im / aa) : cx<T>(T(1), T(0));
    }
    __syncthreads();
    if (tid == 0) {
      cx<T> dcur(T(1), T(0));
      Dp[0] = dcur;
      for (int c = 0; c + 1 < n; ++c) {
        dcur = dcur * al[c];
        Dp[c + 1] = dcur;
      }
      od[n - 1] = T(0);
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Stage 2, lower-triangle form (used when its shared memory fits, see the launcher).
// Same reflectors and T' as k_lg_tridiag, one pass over the trailing lower triangle
// per column: the column c+1 of the updated matrix is formed first, its reflector
// u' built, and then the rank-2 update of step c and the product p' = A' u' of step
// c+1 run in the same sweep.  A' u' takes A'_rq u'_q from the stored lower triangle
// and conj(A'_rq) u'_r for the mirrored upper one; the mirrored terms go to one
// accumulator array per warp (lane-private entries: entry q of a warp's array is
// only touched by lane (q - lo) mod 32), summed over warps in a fixed order, so the
// result does not depend on scheduling.
// ---------------------------------------------------------------------------

// Block-wide sum in the working precision (FP32 for the mixed solve: GB300's FP64
// pipe is ~70x narrower, and these per-step reductions would otherwise cost as much
// as the sweep over the matrix), with one barrier: the caller's next use of `red` comes
// after another one.
template <typename T>
__device__ __forceinline__ T block_sum_1(T v, T* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  T s = T(0);
  for (int k = 0; k < int(blockDim.x >> 5); ++k) s += red[k];
  return s;
}

// The reflector of a column x with leading entry x0 and |x|^2 - |x0|^2 = tail: (I - 2 u u^dag) x =
// alpha e_1 with u = inv (x - alpha e_1), u_0 = inv v0; u = 0 and alpha = x0 when nothing
// lies below the leading entry.
template <typename T>
struct LgReflector {
  cx<T> alpha, v0;
  T inv;
  __device__ LgReflector(cx<T> x0, T tail) : alpha(x0), v0(T(0), T(0)), inv(T(0)) {
    if (!(tail > T(0))) return;
    const T ax2 = abs2(x0), ax0 = sqrt(ax2), nx = sqrt(ax2 + tail);
    const cx<T> ph = ax0 > T(0) ? cx<T>(x0.re / ax0, x0.im / ax0) : cx<T>(T(1), T(0));
    const T v0m = ax0 + nx;
    inv = T(1) / sqrt(v0m * v0m + tail);
    v0 = v0m * ph;
    alpha = -nx * ph;
  }
};

// Rows and columns lo..n-1 of the lower triangle: with upd, A <- A - 2 (u w^dag + w u^dag);
// then A u2 into pw (per-warp accumulators, stride n).  A warp takes RW rows at a
// time (r, r + nwarp, ...) and walks their columns together, so that RW loads per
// lane are in flight even when the rows are short.  Row r is read at src(r)[q] and, with upd
// or kCopy, written to dst(r)[q].  The caller zeroes pw before and sums it over warps after.
template <typename T, bool kCopy, class SR, class DR>
__device__ void lg_hpass(SR src, DR dst, int n, int lo, bool upd, const cx<T>* u, const cx<T>* w,
                         const cx<T>* u2, cx<T>* pw) {
  constexpr int RW = sizeof(T) == 4 ? 8 : 4;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  cx<T>* acc_w = pw + warp * n;
  const cx<T> zero(T(0), T(0));
  for (int r0 = lo + warp; r0 < n; r0 += RW * nwarp) {
    int rr[RW];
    cx<T> ur[RW], wr[RW], u2r[RW], acc[RW];
    int rmax = r0;
#pragma unroll
    for (int i = 0; i < RW; ++i) {
      rr[i] = r0 + i * nwarp;
      const bool ok = rr[i] < n;
      if (ok) rmax = rr[i];
      ur[i] = ok && upd ? T(2) * u[rr[i]] : zero;
      wr[i] = ok && upd ? T(2) * w[rr[i]] : zero;
      u2r[i] = ok ? u2[rr[i]] : zero;
      acc[i] = zero;
      if (!ok) rr[i] = -1;
    }
    for (int q = lo + lane; q <= rmax; q += 32) {
      cx<T> v[RW];
#pragma unroll
      for (int i = 0; i < RW; ++i)
        v[i] = q <= rr[i] ? src(rr[i])[q] : zero;
      const cx<T> wq = upd ? w[q] : zero, uq = upd ? u[q] : zero, u2q = u2[q];
      cx<T> tq = zero;
#pragma unroll
      for (int i = 0; i < RW; ++i) {
        if (q > rr[i]) continue;
        cx<T> x = v[i];
        if (upd) {
          // FP64: eight fused operations.  FP32, where latency counts: the two products side by
          // side (n = 400, 256 k-points: 12.1 ms against 15.2 with the fused chain)
          if constexpr (sizeof(T) == 8) {
            cfms(x, ur[i], conj(wq));
            cfms(x, wr[i], conj(uq));
          } else {
            x = x - (ur[i] * conj(wq) + wr[i] * conj(uq));
          }
          if (q == rr[i]) x.im = T(0);
        }
        if (upd || kCopy) dst(rr[i])[q] = x;
        cfma(acc[i], x, u2q);
        if (q < rr[i]) {
          if constexpr (sizeof(T) == 8)
            cfma_conj(tq, x, u2r[i]);
          else
            tq = tq + conj(x) * u2r[i];
        }
      }
      acc_w[q] = acc_w[q] + tq;
    }
#pragma unroll
    for (int i = 0; i < RW; ++i) {
      const cx<T> t = warp_csum(acc[i]);
      // entry r belongs to lane (r - lo) mod 32 of this warp's array
      if (rr[i] >= 0 && lane == ((rr[i] - lo) & 31)) acc_w[rr[i]] = acc_w[rr[i]] + t;
    }
    __syncwarp();
  }
}

// kShared: the matrix is held in shared memory (packed lower triangle) from the first sweep on.
// A step has five block barriers: the column with its norm, the reflector, the sweep, p = A u
// with u^dag p, and w.
template <typename T, bool kShared>
__global__ void __launch_bounds__(512) k_lg_tridiag_h(LargeArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int n = a.n, tid = threadIdx.x, nt = blockDim.x, nwarp = nt >> 5;
  cx<T>* u = reinterpret_cast<cx<T>*>(smem);  // reflector of the current step
  cx<T>* w = u + n;
  cx<T>* u2 = w + n;                          // reflector of the next step
  cx<T>* pa = u2 + n;                         // A u2
  cx<T>* al = pa + n;                         // complex subdiagonal
  cx<T>* pw = al + n;                         // (blockDim / 32) x n per-warp accumulators
  T* red = reinterpret_cast<T*>(pw + nwarp * n);  // two buffers of 16 partial sums, x0
  cx<T>* x0s = reinterpret_cast<cx<T>*>(red + 32);
  cx<T>* tri = reinterpret_cast<cx<T>*>(reinterpret_cast<double*>(red) + 64);
  for (long long kw = blockIdx.x; kw < a.W; kw += gridDim.x) {
    if (std::is_same<T, double>::value && a.need && !a.need[kw]) continue;
    cx<T>* A = reinterpret_cast<cx<T>*>(a.A) + kw * (long long)n * n;
    T* dg = reinterpret_cast<T*>(a.dg) + kw * n;
    T* od = reinterpret_cast<T*>(a.od) + kw * n;
    cx<T>* Dp = reinterpret_cast<cx<T>*>(a.Dp) + kw * n;
    auto grow = [&](int r) { return A + (long long)r * n; };
    auto trow = [&](int r) { return kShared ? tri + r * (r + 1) / 2 : grow(r); };
    // the column in u2[lo..n) with the partial sum s of its tail becomes the reflector, which
    // also goes to column lo - 1 of A
    auto reflect = [&](T s, int lo) {
      s = block_sum_1(s, red);
      const LgReflector<T> f(*x0s, s);
      if (tid == 0) al[lo - 1] = f.alpha;
      for (int r = lo + tid; r < n; r += nt) {
        const cx<T> v = f.inv * (r == lo ? f.v0 : u2[r]);
        u2[r] = v;
        grow(r)[lo - 1] = v;
      }
      __syncthreads();
    };
    // after a sweep: pa = A u2, w = pa - (u2^dag pa) u2; u2 becomes u
    auto finish = [&](int lo) {
      __syncthreads();
      T kr = T(0);
      for (int q = lo + tid; q < n; q += nt) {
        cx<T> t(T(0), T(0));
        for (int k = 0; k < nwarp; ++k) {
          t = t + pw[k * n + q];
          pw[k * n + q] = cx<T>(T(0), T(0));
        }
        pa[q] = t;
        kr += u2[q].re * t.re + u2[q].im * t.im;
      }
      kr = block_sum_1(kr, red + 16);
      for (int q = lo + tid; q < n; q += nt) w[q] = pa[q] - kr * u2[q];
      cx<T>* t = u;
      u = u2;
      u2 = t;
      __syncthreads();
    };
    // step 0: reflector of column 0 and p = A22 u
    for (int e = tid; e < nwarp * n; e += nt) pw[e] = cx<T>(T(0), T(0));
    T s = T(0);
    for (int r = 1 + tid; r < n; r += nt) {
      const cx<T> x = A[(long long)r * n];
      u2[r] = x;
      if (r == 1)
        *x0s = x;
      else
        s += abs2(x);
    }
    if (tid == 0) dg[0] = A[0].re;
    reflect(s, 1);
    lg_hpass<T, kShared>(grow, trow, n, 1, false, nullptr, nullptr, u2, pw);
    finish(1);
    if (n == 2 && tid == 0) dg[1] = trow(1)[1].re;
    for (int c = 0; c + 2 < n; ++c) {
      // column c+1 of A - 2 (u w^dag + w u^dag), rows c+1..n-1
      const cx<T> uc = T(2) * conj(u[c + 1]), wc = T(2) * conj(w[c + 1]);
      s = T(0);
      for (int r = c + 1 + tid; r < n; r += nt) {
        cx<T> x = trow(r)[c + 1];
        cfms(x, u[r], wc);
        cfms(x, w[r], uc);
        u2[r] = x;
        if (r == c + 1)
          dg[c + 1] = x.re;
        else if (r == c + 2)
          *x0s = x;
        else
          s += abs2(x);
      }
      if (c + 3 == n) {  // last 2 x 2 block: its subdiagonal and diagonal, no reflector
        __syncthreads();
        if (tid == 0) {
          al[n - 2] = u2[n - 1];
          const cx<T> un = u[n - 1], wn = w[n - 1];
          dg[n - 1] = trow(n - 1)[n - 1].re - T(4) * (un.re * wn.re + un.im * wn.im);
          A[(long long)(n - 1) * n + n - 2] = cx<T>(T(0), T(0));
        }
        __syncthreads();
        break;
      }
      reflect(s, c + 2);
      lg_hpass<T, false>(trow, trow, n, c + 2, true, u, w, u2, pw);
      finish(c + 2);
    }
    // unit phases of the subdiagonal, then their prefix products (serial: cheap)
    for (int c = tid; c + 1 < n; c += nt) {
      const T aa = sqrt(abs2(al[c]));
      od[c] = aa;
      al[c] = aa > T(0) ? cx<T>(al[c].re / aa, al[c].im / aa) : cx<T>(T(1), T(0));
    }
    __syncthreads();
    if (tid == 0) {
      cx<T> dcur(T(1), T(0));
      Dp[0] = dcur;
      for (int c = 0; c + 1 < n; ++c) {
        dcur = dcur * al[c];
        Dp[c + 1] = dcur;
      }
      od[n - 1] = T(0);
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Stage 3: eigenvalues of T' by bisection on Sturm counts, one thread per
// (k-point, eigenvalue index), T' of one k-point in the CTA's shared memory.
//
// The count at x is the number of sign changes of the leading principal minors
//   p_{i+1} = (d_i - x) p_i - e_{i-1}^2 p_{i-1}
// (Givens), rescaled by a power of two every few rows.  The ratios q_i = p_{i+1} / p_i need
// a division per row on the critical path (~1400 clocks in FP64, ~60 in FP32) where the
// minors need one fused multiply-add (64, 4.5).  An FP64 bisection starts from the FP32 one
// (a bracket 2e-5 ||T'|| wide, checked by FP64 counts and widened where it does not hold).
// Measured, with the spin operator's eigensolves: n = 124 FP64, 256 k-points, 6.1 -> 1.9 ms;
// n = 324 mixed, 36 k-points, 5.5 -> 1.7 ms; n = 256 FP32, 837 k-points, 1.2 -> 0.57 ms.
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void gershgorin(const T* dg, const T* od, int n, T& lo, T& hi, T& tn) {
  lo = T(INFINITY);
  hi = -T(INFINITY);
  tn = T(0);
  for (int i = 0; i < n; ++i) {
    const T r = (i > 0 ? od[i - 1] : T(0)) + (i + 1 < n ? od[i] : T(0));
    lo = fmin(lo, dg[i] - r);
    hi = fmax(hi, dg[i] + r);
    tn = fmax(tn, fabs(dg[i]) + r);
  }
}

// 2^-e for |x| in [2^e, 2^(e+1)), from the exponent bits (x normal or zero).
__device__ __forceinline__ float pow2_inv(float x) {
  return __int_as_float(0x7f000000 - (__float_as_int(x) & 0x7f800000));
}
__device__ __forceinline__ double pow2_inv(double x) {
  return __hiloint2double(0x7fe00000 - (__double2hiint(x) & 0x7ff00000), 0);
}

// Sturm count at x of the scaled matrix (entries of T' / ||T'||, |d|, |e| <= 1): d and e2 =
// e_{i-1}^2 per row (e2[0] = 0), padded to a multiple of UN rows with d = 4, e2 = 0 (no sign
// change for x < 4).  Between two rescalings a minor loses at most a factor
// (min(1e-12, e2))^UN, inside the exponent range.
template <typename T>
__device__ __forceinline__ int sturm_count(const T* d, const T* e2, int npad, T x) {
  constexpr int UN = sizeof(T) == 4 ? 2 : 8;
  T pm = T(0), pc = T(1);
  int cnt = 0;
  for (int i = 0; i < npad; i += UN) {
#pragma unroll
    for (int u = 0; u < UN; ++u) {
      T pn = fma(d[i + u] - x, pc, -(e2[i + u] * pm));
      if (pn == T(0)) pn = T(-1e-12) * pc;  // a zero minor counts as a change of sign
      cnt += signbit(pn) != signbit(pc);
      pm = pc;
      pc = pn;
    }
    const T s = pow2_inv(fmax(fabs(pm), fabs(pc)));
    pm *= s;
    pc *= s;
  }
  return cnt;
}

constexpr int BIS_THREADS = 128;

__host__ __device__ inline int bisect_pad(int n) { return (n + 7) & ~7; }

template <typename T>
__host__ __device__ inline size_t bisect_smem(int n) {
  return size_t(bisect_pad(n)) * 2 * (sizeof(T) + (sizeof(T) == 8 ? sizeof(float) : 0));
}

// Bisection for eigenvalue idx of the scaled matrix from a bracket lo < hi, to 2 eps |lambda|
// or an eighth of eps ||T'||.
template <typename T>
__device__ __forceinline__ void bisect_run(const T* d, const T* e2, int npad, int idx, T& lo, T& hi) {
  for (int it = 0; it < 96; ++it) {
    const T mid = T(0.5) * (lo + hi);
    if (!(mid > lo && mid < hi)) break;
    if (hi - lo <= T(2) * lg_eps<T>() * fmax(T(0.0625), fmax(fabs(lo), fabs(hi)))) break;
    if (sturm_count(d, e2, npad, mid) > idx)
      hi = mid;
    else
      lo = mid;
  }
}

template <typename T>
__global__ void __launch_bounds__(BIS_THREADS) k_lg_bisect(LargeArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr bool k64 = sizeof(T) == 8;
  const int n = a.n, tid = threadIdx.x, np = bisect_pad(n);
  T* d = reinterpret_cast<T*>(smem);
  T* e2 = d + np;
  float* df = reinterpret_cast<float*>(e2 + np);  // FP64: the matrix in FP32 as well
  float* ef = df + np;
  __shared__ T rlo[BIS_THREADS / 32], rhi[BIS_THREADS / 32], rtn[BIS_THREADS / 32];
  for (long long kw = blockIdx.x; kw < a.W; kw += gridDim.x) {
    if (std::is_same<T, double>::value && a.need && !a.need[kw]) continue;
    const T* dg = reinterpret_cast<const T*>(a.dg) + kw * n;
    const T* od = reinterpret_cast<const T*>(a.od) + kw * n;
    // Gershgorin interval and ||T'||
    T lo = T(INFINITY), hi = -T(INFINITY), tn = T(0);
    for (int i = tid; i < n; i += BIS_THREADS) {
      const T di = dg[i], r = (i > 0 ? od[i - 1] : T(0)) + (i + 1 < n ? od[i] : T(0));
      lo = fmin(lo, di - r);
      hi = fmax(hi, di + r);
      tn = fmax(tn, fabs(di) + r);
    }
    for (int o = 16; o > 0; o >>= 1) {
      lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
      tn = fmax(tn, __shfl_xor_sync(0xffffffffu, tn, o));
    }
    __syncthreads();
    if ((tid & 31) == 0) {
      rlo[tid >> 5] = lo;
      rhi[tid >> 5] = hi;
      rtn[tid >> 5] = tn;
    }
    __syncthreads();
    for (int w = 0; w < BIS_THREADS / 32; ++w) {
      lo = fmin(lo, rlo[w]);
      hi = fmax(hi, rhi[w]);
      tn = fmax(tn, rtn[w]);
    }
    // scaled by a power of two (exact): |entries| <= 1
    const T tnc = fmax(tn, T(1e-30)), sc = T(0.5) * pow2_inv(tnc);
    for (int i = tid; i < np; i += BIS_THREADS) {
      const T di = i < n ? dg[i] * sc : T(4), ei = i > 0 && i < n ? od[i - 1] * sc : T(0);
      d[i] = di;
      e2[i] = ei * ei;
      if constexpr (k64) {
        df[i] = float(di);
        ef[i] = float(ei) * float(ei);
      }
    }
    __syncthreads();
    lo *= sc;
    hi *= sc;
    const T span = fmax(hi - lo, T(1e-30));
    lo -= T(4) * lg_eps<T>() * span + T(1e-30);
    hi += T(4) * lg_eps<T>() * span + T(1e-30);
    for (int idx = blockIdx.y * BIS_THREADS + tid; idx < a.nval; idx += gridDim.y * BIS_THREADS) {
      T l = lo, h = hi;
      if constexpr (k64) {
        float fl = float(lo) - 1e-6f, fh = float(hi) + 1e-6f;
        bisect_run<float>(df, ef, np, idx, fl, fh);
        T w = T(1e-5);
        for (; w < T(8); w *= T(64)) {
          l = fmax(lo, T(fl) - w);
          h = fmin(hi, T(fh) + w);
          if (sturm_count(d, e2, np, l) <= idx && sturm_count(d, e2, np, h) > idx) break;
        }
        if (!(w < T(8))) {
          l = lo;
          h = hi;
        }
      }
      bisect_run<T>(d, e2, np, idx, l, h);
      reinterpret_cast<T*>(a.lam)[kw * a.nval + idx] = T(0.5) * (l + h) / sc;
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Stage 4: eigenvectors of T' by inverse iteration.  (T' - lambda) = P L U with
// partial pivoting (U has two superdiagonals); three solves from a fixed
// pseudo-random start.  Eigenvalues closer than 1e-3 ||T'|| form a cluster, whose
// vectors one thread computes in order, orthogonalising each against the earlier
// ones of its cluster at every iteration.  Above INVIT_WINDOW_N, where the spectrum
// of a supercell is so dense that the chained clusters span most of it, a vector is
// orthogonalised only against the earlier ones within 1e-3 ||T'|| of its eigenvalue:
// two vectors further apart are orthogonal to ~eps ||T'|| / (1e-3 ||T'||) already, the
// bound the cluster rule accepts between clusters, and the cost per vector is O(n)
// instead of O(n x cluster size).
// Where only the span of the computed vectors matters (subspace_only: the PSO
// sector), every vector iterates on its own thread at once instead, converging into
// its cluster's invariant subspace from a distinct start, and a second kernel
// orthonormalises each cluster's vectors by modified Gram-Schmidt applied twice,
// one warp per cluster: a cluster of p/2 exactly degenerate PSO eigenvalues no
// longer serialises on one thread.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double hash_unit(unsigned long long x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  x ^= x >> 31;
  return double(x >> 11) * (1.0 / 9007199254740992.0) * 2.0 - 1.0;
}

// Interleaved per-thread arrays: element r of thread t's array a lives at
// base[(a * n + r) * NT + t], so a warp's accesses to the same r are contiguous.
template <typename T>
struct Strided {
  T* base;
  long long NT;
  int n;
  __device__ __forceinline__ T& at(int a, int r, long long t) const { return base[((long long)a * n + r) * NT + t]; }
};

// Rows whose operands are loaded together: the recurrences below are serial, but their
// operands (interleaved global memory, an L2 or DRAM round trip each) do not depend on them.
// n = 400, 256 k-points, all vectors: 17.5 -> 8.0 ms (with the reciprocal pivots kept).
constexpr int TRI_U = 8;

template <typename T>
__device__ void tri_factor(const T* dg, const T* od, int n, T lam, T tiny, const Strided<T>& W,
                           long long t) {
  T c0 = dg[0] - lam, c1 = n > 1 ? od[0] : T(0);
  auto pivot = [&](T d) {  // what the solves multiply by
    if (fabs(d) < tiny) d = d < T(0) ? -tiny : tiny;
    return T(1) / d;
  };
  for (int i = 0; i + 1 < n; ++i) {
    const T b = od[i];                          // subdiagonal entry of row i+1
    const T a1 = dg[i + 1] - lam;               // diagonal of row i+1
    const T e1 = i + 2 < n ? od[i + 1] : T(0);  // superdiagonal of row i+1
    if (fabs(b) > fabs(c0)) {                   // swap rows i and i+1
      const T r = T(1) / b, m = c0 * r;
      W.at(0, i, t) = fabs(b) < tiny ? pivot(b) : r; W.at(1, i, t) = a1; W.at(2, i, t) = e1;
      W.at(3, i, t) = m; W.at(4, i, t) = T(1);
      const T r1 = c1 - m * a1, r2 = -m * e1;   // remaining row: columns i+1, i+2
      c0 = r1; c1 = r2;
    } else {
      if (c0 == T(0)) c0 = tiny;
      const T r = T(1) / c0, m = b * r;
      W.at(0, i, t) = fabs(c0) < tiny ? pivot(c0) : r; W.at(1, i, t) = c1; W.at(2, i, t) = T(0);
      W.at(3, i, t) = m; W.at(4, i, t) = T(0);
      c0 = a1 - m * c1;
      c1 = e1;
    }
  }
  W.at(0, n - 1, t) = pivot(c0);
  W.at(1, n - 1, t) = T(0);
  W.at(2, n - 1, t) = T(0);
}

// Solves (T' - lambda) x = b in place on array 5 of the thread's scratch.
template <typename T>
__device__ void tri_solve(int n, const Strided<T>& W, long long t) {
  T xi = W.at(5, 0, t);
  for (int i0 = 0; i0 + 1 < n; i0 += TRI_U) {
    T xn[TRI_U], m[TRI_U], sw[TRI_U];
#pragma unroll
    for (int u = 0; u < TRI_U; ++u) {
      const int i = i0 + u;
      const bool in = i + 1 < n;
      xn[u] = in ? W.at(5, i + 1, t) : T(0);
      m[u] = in ? W.at(3, i, t) : T(0);
      sw[u] = in ? W.at(4, i, t) : T(0);
    }
#pragma unroll
    for (int u = 0; u < TRI_U; ++u) {
      const int i = i0 + u;
      if (i + 1 >= n) break;
      T x = xn[u];
      if (sw[u] != T(0)) { const T q = xi; xi = x; x = q; }
      W.at(5, i, t) = xi;
      xi = x - m[u] * xi;
    }
  }
  W.at(5, n - 1, t) = xi;
  T x1 = T(0), x2 = T(0);  // x_{i+1}, x_{i+2}
  for (int i0 = n - 1; i0 >= 0; i0 -= TRI_U) {
    T b[TRI_U], r[TRI_U], u1[TRI_U], u2[TRI_U];
#pragma unroll
    for (int u = 0; u < TRI_U; ++u) {
      const int i = i0 - u;
      const bool in = i >= 0;
      b[u] = in ? W.at(5, i, t) : T(0);
      r[u] = in ? W.at(0, i, t) : T(0);
      u1[u] = in ? W.at(1, i, t) : T(0);
      u2[u] = in ? W.at(2, i, t) : T(0);
    }
#pragma unroll
    for (int u = 0; u < TRI_U; ++u) {
      const int i = i0 - u;
      if (i < 0) break;
      const T x = (b[u] - u1[u] * x1 - u2[u] * x2) * r[u];
      W.at(5, i, t) = x;
      x2 = x1;
      x1 = x;
    }
  }
}

// x (array 5) scaled to unit norm; with Zc, also written to the vector's column of Z.
template <typename T>
__device__ void tri_normalise(int n, const Strided<T>& W, long long t, T* Zc, int nv) {
  T s2 = T(0);
#pragma unroll 8
  for (int r = 0; r < n; ++r) {
    const T x = W.at(5, r, t);
    s2 += x * x;
  }
  s2 = T(1) / sqrt(s2);
  for (int r0 = 0; r0 < n; r0 += TRI_U) {
    T x[TRI_U];
#pragma unroll
    for (int u = 0; u < TRI_U; ++u) x[u] = r0 + u < n ? s2 * W.at(5, r0 + u, t) : T(0);
#pragma unroll
    for (int u = 0; u < TRI_U; ++u)
      if (r0 + u < n) {
        if (Zc)
          Zc[(long long)(r0 + u) * nv] = x[u];
        else
          W.at(5, r0 + u, t) = x[u];
      }
  }
}

// What a stage after the eigenvalues skips: the FP32 ones the k-points that the polish cannot
// take, the FP64 ones the others.
template <typename T>
__device__ __forceinline__ bool lg_skip(const LargeArgs& a, long long kw) {
  return a.need && (a.need[kw] != 0) == (sizeof(T) == 4);
}

constexpr int INVIT_WINDOW_N = 512, INVIT_ITS = 3;

template <typename T>
__global__ void k_lg_invit(LargeArgs a) {
  const long long NT = a.W * a.nvec;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= NT) return;
  const long long kw = t / a.nvec;
  if (lg_skip<T>(a, kw)) return;
  const int idx = int(t - kw * a.nvec), n = a.n, nv = a.nvec;
  const T* dg = reinterpret_cast<const T*>(a.dg) + kw * n;
  const T* od = reinterpret_cast<const T*>(a.od) + kw * n;
  const T* lam = reinterpret_cast<const T*>(a.lam) + kw * a.nval;
  T lo, hi, tn;
  gershgorin(dg, od, n, lo, hi, tn);
  const T tolc = T(1e-3) * tn;
  if (idx > 0 && lam[idx] - lam[idx - 1] <= tolc) return;  // not the first of its cluster
  int end = idx;
  while (end + 1 < nv && lam[end + 1] - lam[end] <= tolc) ++end;
  T* Z = reinterpret_cast<T*>(a.Z) + kw * (long long)nv * n;   // row-major n x nvec
  const Strided<T> W{reinterpret_cast<T*>(a.work), NT, n};
  const T tiny = fmax(lg_eps<T>() * tn, T(1e-30));
  const bool windowed = n > INVIT_WINDOW_N;
  int q0 = idx;  // first earlier vector of the cluster to orthogonalise against
  for (int j = idx; j <= end; ++j) {
    if (windowed)
      while (lam[j] - lam[q0] > tolc) ++q0;
    tri_factor(dg, od, n, lam[j], tiny, W, t);
    for (int r = 0; r < n; ++r) W.at(5, r, t) = T(hash_unit((unsigned long long)j * 1000003ull + r));
    for (int it = 0; it < INVIT_ITS; ++it) {
      tri_solve(n, W, t);
      for (int q = q0; q < j; ++q) {  // orthogonalise within the cluster (or its window)
        T d = T(0);
#pragma unroll 8
        for (int r = 0; r < n; ++r) d += Z[(long long)r * nv + q] * W.at(5, r, t);
        for (int r0 = 0; r0 < n; r0 += TRI_U) {
          T x[TRI_U];
#pragma unroll
          for (int u = 0; u < TRI_U; ++u)
            x[u] = r0 + u < n ? W.at(5, r0 + u, t) - d * Z[(long long)(r0 + u) * nv + q] : T(0);
#pragma unroll
          for (int u = 0; u < TRI_U; ++u)
            if (r0 + u < n) W.at(5, r0 + u, t) = x[u];
        }
      }
      tri_normalise(n, W, t, it + 1 == INVIT_ITS ? Z + j : static_cast<T*>(nullptr), nv);
    }
  }
}

template <typename T>
__global__ void k_lg_invit_par(LargeArgs a) {
  const long long NT = a.W * a.nvec;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= NT) return;
  const long long kw = t / a.nvec;
  const int j = int(t - kw * a.nvec), n = a.n, nv = a.nvec;
  const T* dg = reinterpret_cast<const T*>(a.dg) + kw * n;
  const T* od = reinterpret_cast<const T*>(a.od) + kw * n;
  const T* lam = reinterpret_cast<const T*>(a.lam) + kw * a.nval;
  T lo, hi, tn;
  gershgorin(dg, od, n, lo, hi, tn);
  T* Z = reinterpret_cast<T*>(a.Z) + kw * (long long)nv * n;   // row-major n x nvec
  const Strided<T> W{reinterpret_cast<T*>(a.work), NT, n};
  const T tiny = fmax(lg_eps<T>() * tn, T(1e-30));
  tri_factor(dg, od, n, lam[j], tiny, W, t);
  for (int r = 0; r < n; ++r) W.at(5, r, t) = T(hash_unit((unsigned long long)j * 1000003ull + r));
  for (int it = 0; it < INVIT_ITS; ++it) {
    tri_solve(n, W, t);
    tri_normalise(n, W, t, it + 1 == INVIT_ITS ? Z + j : static_cast<T*>(nullptr), nv);
  }
}

// Orthonormalises the vectors of each cluster in place: one warp per eigenvalue index,
// working only where the index starts a cluster of two or more.
template <typename T>
__global__ void k_lg_invit_orth(LargeArgs a) {
  const long long NT = a.W * a.nvec;
  const long long t = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (t >= NT) return;
  const long long kw = t / a.nvec;
  const int idx = int(t - kw * a.nvec), n = a.n, nv = a.nvec;
  const T* dg = reinterpret_cast<const T*>(a.dg) + kw * n;
  const T* od = reinterpret_cast<const T*>(a.od) + kw * n;
  const T* lam = reinterpret_cast<const T*>(a.lam) + kw * a.nval;
  T lo, hi, tn;
  gershgorin(dg, od, n, lo, hi, tn);
  const T tolc = T(1e-3) * tn;
  if (idx > 0 && lam[idx] - lam[idx - 1] <= tolc) return;  // not the first of its cluster
  int end = idx;
  while (end + 1 < nv && lam[end + 1] - lam[end] <= tolc) ++end;
  if (end == idx) return;
  T* Z = reinterpret_cast<T*>(a.Z) + kw * (long long)nv * n;
  for (int j = idx; j <= end; ++j) {
    for (int pass = 0; pass < 2; ++pass)
      for (int q = idx; q < j; ++q) {
        T d = T(0);
        for (int r = lane; r < n; r += 32) d += Z[(long long)r * nv + q] * Z[(long long)r * nv + j];
        for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
        for (int r = lane; r < n; r += 32) Z[(long long)r * nv + j] -= d * Z[(long long)r * nv + q];
      }
    T s2 = T(0);
    for (int r = lane; r < n; r += 32) s2 += Z[(long long)r * nv + j] * Z[(long long)r * nv + j];
    for (int o = 16; o > 0; o >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    s2 = T(1) / sqrt(s2);
    for (int r = lane; r < n; r += 32) Z[(long long)r * nv + j] *= s2;
  }
}

// Levels of T' within 1e-3 of the spectral radius of the upper edge p (lam ascending, all n).
__device__ __forceinline__ float polish_width(const float* lam, int n) {
  return 1e-3f * fmaxf(fabsf(lam[0]), fabsf(lam[n - 1]));
}
__device__ __forceinline__ int polish_upper(const float* lam, int n, int p) {
  const float w = polish_width(lam, n);
  int c = p;
  while (c + 1 < n && c - p < POLISH_G && lam[c + 1] - lam[p] <= w) ++c;
  return c - p + 1;
}
__device__ __forceinline__ int polish_lower(const float* lam, int n, int p) {
  const float w = polish_width(lam, n);
  int c = p - 1;
  while (c > 0 && p - c <= POLISH_G && lam[p - 1] - lam[c - 1] <= w) --c;
  return p - c;
}

// Which k-points the polish can take, from the FP32 eigenvalues: energies in range, a gap of 1e-3
// of the spectral radius, band edges of at most POLISH_G levels.  Told before the eigenvectors,
// so that a k-point left to the FP64 solve costs the FP32 reduction and bisection only.
// Where that is a quarter of the wave or more, the whole wave is left to it: the two solves are
// chains of the same length whatever the number of their k-points, and would follow each other.
// One CTA.
__global__ void __launch_bounds__(256) k_lg_polish_need(LargeArgs a) {
  __shared__ double red[32];
  double left = 0.0;
  for (long long kw = threadIdx.x; kw < a.W; kw += blockDim.x) {
    const float* lam = reinterpret_cast<const float*>(a.lam) + kw * a.nval;
    const float width = polish_width(lam, a.n), nrm = 1e3f * width;
    const bool fit = nrm > 1e-8f && nrm < 1e12f && lam[a.p] - lam[a.p - 1] > width &&
                     polish_upper(lam, a.n, a.p) <= POLISH_G && polish_lower(lam, a.n, a.p) <= POLISH_G;
    a.need[kw] = fit ? 0 : 1;
    left += fit ? 0.0 : 1.0;
  }
  if (4.0 * block_sum(left, red) < double(a.W)) return;
  for (long long kw = threadIdx.x; kw < a.W; kw += blockDim.x) a.need[kw] = 1;
}

// ---------------------------------------------------------------------------
// Stage 5: back-transform x = Q D z for the first ncol eigenvectors, Q = P_0 ... P_{n-3}:
// X = D Z, then X <- P_c X for c = n-3 down to 0 (P_c = I - 2 u_c u_c^dagger): one
// reflector at a time in FP64, in blocks of 32 reflectors (compact WY form) in FP32.
// Output X[r][col] with leading dimension ncol, precision To.
// ---------------------------------------------------------------------------
template <typename T, typename To>
__global__ void __launch_bounds__(256, 2) k_lg_backtransform(LargeArgs a, cx<To>* out, long long out_stride,
                                                             int ncol, int pw) {
  static_assert(std::is_same<T, To>::value, "the back-transform keeps the solver's precision");
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr bool kTc = std::is_same<T, float>::value;  // FP32: compact WY on the tensor cores
  __shared__ uint32_t tmem_slot;
  __shared__ __align__(8) uint64_t tc_bar;
  tc::State ts{};
  if constexpr (kTc) ts = tc::setup(&tmem_slot, &tc_bar);
  const int n = a.n, tid = threadIdx.x, nt = blockDim.x;
  for (long long kw = blockIdx.x; kw < a.W; kw += gridDim.x) {
    if (lg_skip<T>(a, kw)) continue;
    const cx<T>* A = reinterpret_cast<const cx<T>*>(a.A) + kw * (long long)n * n;
    const cx<T>* Dp = reinterpret_cast<const cx<T>*>(a.Dp) + kw * n;
    const T* Z = reinterpret_cast<const T*>(a.Z) + kw * (long long)a.nvec * n;
    cx<To>* X = out + kw * out_stride;
    int nc = ncol;  // columns of this k-point (the polish: the occupied ones and the upper edge's)
    if constexpr (kTc)
      if (a.polish)
        nc = min(ncol, a.p + polish_upper(reinterpret_cast<const float*>(a.lam) + kw * a.nval, n, a.p));
    for (int r = tid >> 5; r < n; r += nt >> 5) {
      const cx<T> d = Dp[r];
      for (int col = tid & 31; col < nc; col += 32) {
        const T z = Z[(long long)r * a.nvec + col];
        X[(long long)r * ncol + col] = cx<To>(To(d.re * z), To(d.im * z));
      }
    }
    __syncthreads();
    if constexpr (!kTc) {
      cta_reflect<T, To>(A, n, X, ncol, ncol, true, smem, pw);   // FP64-pipe bound: fewest flops
    } else if (!ts.failed) {                                     // blocked, tensor-core GEMMs
      if (!cta_reflect_wy(A, n, X, nc, ncol, true, smem, ts) && tid == 0)
        report(a.status, ST_ETIMEOUT, a.k0 + kw, 0.0);
    }
  }
  if constexpr (kTc) tc::teardown(ts);
}

// FP64 back-transform for large n (a one-reflector panel would hold fewer than 16
// columns): X = D Z, then the reflectors in compact-WY blocks through FP64 GEMMs.
__global__ void __launch_bounds__(256, 2) k_lg_backtransform_wy64(LargeArgs a, z64* out, long long out_stride,
                                                                  int ncol) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int n = a.n, tid = threadIdx.x, nt = blockDim.x;
  for (long long kw = blockIdx.x; kw < a.W; kw += gridDim.x) {
    if (a.need && !a.need[kw]) continue;
    const z64* A = reinterpret_cast<const z64*>(a.A) + kw * (long long)n * n;
    const z64* Dp = reinterpret_cast<const z64*>(a.Dp) + kw * n;
    const double* Z = reinterpret_cast<const double*>(a.Z) + kw * (long long)a.nvec * n;
    z64* X = out + kw * out_stride;
    for (int r = tid >> 5; r < n; r += nt >> 5) {
      const z64 d = Dp[r];
      for (int col = tid & 31; col < ncol; col += 32) {
        const double z = Z[(long long)r * a.nvec + col];
        X[(long long)r * ncol + col] = z64(d.re * z, d.im * z);
      }
    }
    __syncthreads();
    cta_reflect_wy_simt<double>(A, n, X, ncol, ncol, true, smem);
  }
}

// FP64 path: direct gap from the bisection eigenvalues.
__global__ void k_lg_gap64(LargeArgs a) {
  const long long kw = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (kw >= a.W || (a.need && !a.need[kw])) return;
  const double* lam = reinterpret_cast<const double*>(a.lam) + kw * a.nval;
  const double g = a.p < a.n ? lam[a.p] - lam[a.p - 1] : INFINITY;
  const long long k = a.k0 + kw * (a.kstride > 0 ? a.kstride : 1);
  a.gap[k] = g;
  if (!(g > a.gap_tol)) report(a.status, ST_EGAP, k, g);
}

__host__ __device__ inline size_t refine_work_offset(int p) {
  return ((size_t(p) + 66) * sizeof(double) + 15) & ~size_t(15);
}

// ---------------------------------------------------------------------------
// Stage 6 (mixed): one Newton correction of the occupied block.
//   Q = X[:, :p] holds FP32 eigenvectors (exact FP32 numbers).  H Q from the hopping
//   plan's FP64 entries with compensated FP32 dot products; rho_c = q_c^dag H q_c and
//   R = H Q - Q rho in FP64; the complement's coefficients
//   C[a][c] = z_a^T D^dag Q_h^dag R_c / (rho_c - lam_a) and the update
//   Q_h D Z_u C in FP32 through the reflectors (R is small, FP32 keeps it to ~1e-7
//   relative); Q64 = Q + update.  Then one second-order Lowdin step,
//   Q <- Q - Q (E / 2 - 3 E^2 / 8), E = Q^dag Q - I, with Q32^dag Q32 - I compensated and the small
//   terms in FP32.  The gap comes from FP64 Rayleigh quotients of the (p-1)-th
//   and p-th FP32 vectors.  The off-diagonal part of Q^dag H Q is of the order of
//   the FP32 error; its projection on the complement enters at second order.
// ---------------------------------------------------------------------------
// Two CTAs per SM: the compensated GEMM tiles hold 64 accumulator registers per
// thread, and without the bound the kernel takes 136 registers (one CTA per SM).
__global__ void __launch_bounds__(256, 2) k_lg_refine(LargeArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int n = a.n, p = a.p, nbt = a.nbt, tid = threadIdx.x, nt = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nwarp = nt >> 5;
  const DevModel& md = a.model;
  double* rho = reinterpret_cast<double*>(smem);     // p + 2
  double* red = rho + p + 2;                         // 64
  unsigned char* work = smem + refine_work_offset(p);  // block reflectors / GEMM tiles
  __shared__ uint32_t tmem_slot;
  __shared__ __align__(8) uint64_t tc_bar;
  tc::State ts = tc::setup(&tmem_slot, &tc_bar);      // plain FP32 products: tensor cores
  for (long long kw = blockIdx.x; kw < a.W; kw += gridDim.x) {
    if (lg_skip<float>(a, kw)) continue;
    const long long k = a.k0 + kw * (a.kstride > 0 ? a.kstride : 1);
    const c32* A = reinterpret_cast<const c32*>(a.A) + kw * (long long)n * n;
    const c32* Dp = reinterpret_cast<const c32*>(a.Dp) + kw * n;
    const float* Z = reinterpret_cast<const float*>(a.Z) + kw * (long long)a.nvec * n;
    const float* lam = reinterpret_cast<const float*>(a.lam) + kw * a.nval;
    const c32* X = reinterpret_cast<const c32*>(a.X) + kw * (long long)n * nbt;
    const bool dense = a.Hin != nullptr;  // explicit matrix: entries r n + q, all columns
    const z64* He = a.Hent + kw * (long long)(dense ? n * n : md.n_ent);
    z64* Q = a.U + kw * (long long)n * p;
    z64* R = a.R64 + kw * (long long)n * p;          // H Q, later FP32 scratch
    c32* C = a.C32 + kw * (long long)n * p;
    c32* E = reinterpret_cast<c32*>(a.G64 + kw * (long long)p * p);  // Q^dag Q - I (p x p)
    // R = H Q32 (compensated): a tiled GEMM when H is dense, else one warp per row
    if (dense || md.n_ent == n * n) {
      cta_gemm<GemmSplitComp, true, true>(
          n, p, n,
          [&](int r, int q) {
            const c32* hp = reinterpret_cast<const c32*>(He + (long long)r * n + q);
            return SplitC{hp[0], hp[1]};
          },
          [&](int q, int c) { return X[(long long)q * nbt + c]; },
          [&](int r, int c, const CDF& acc) { R[(long long)r * p + c] = acc.value(); }, work);
    } else
    for (int r = warp; r < n; r += nwarp) {
      for (int c0 = 0; c0 < p; c0 += 32) {
        const int c = c0 + lane;
        CDF acc;
        const int q0 = dense ? r * n : a.row_ptr[r], q1 = dense ? (r + 1) * n : a.row_ptr[r + 1];
        for (int q = q0; q < q1; ++q) {
          const c32* hp = reinterpret_cast<const c32*>(He + q);
          const int col = dense ? q - q0 : md.ent_col[q];
          if (c < p) acc.add_prod(hp[0], hp[1], X[(long long)col * nbt + c]);
        }
        if (c < p) R[(long long)r * p + c] = acc.value();
      }
    }
    __syncthreads();
    for (int c = tid; c < p; c += nt) {
      double sum = 0.0;
      for (int r = 0; r < n; ++r) {
        const c32 q = X[(long long)r * nbt + c];
        const z64 h = R[(long long)r * p + c];
        sum += double(q.re) * h.re + double(q.im) * h.im;
      }
      rho[c] = sum;
    }
    __syncthreads();
    // residual to FP32
    for (int r = warp; r < n; r += nwarp)
      for (int c = lane; c < p; c += 32) {
        const z64 h = R[(long long)r * p + c];
        const c32 q = X[(long long)r * nbt + c];
        C[(long long)r * p + c] = c32(float(h.re - rho[c] * double(q.re)), float(h.im - rho[c] * double(q.im)));
      }
    __syncthreads();
    // C <- D^dag Q_h^dag C
    bool tc_ok = cta_reflect_wy(A, n, C, p, p, false, work, ts);
    for (int r = warp; r < n; r += nwarp) {
      const c32 d = conj(Dp[r]);
      for (int c = lane; c < p; c += 32) C[(long long)r * p + c] = d * C[(long long)r * p + c];
    }
    __syncthreads();
    // complement coefficients (FP32), kept in the R workspace
    c32* coef = reinterpret_cast<c32*>(R);
    const int nu = n - p;
    const int nvec = a.nvec;
    // coef[ua][c] = (Z_u^T C)[ua][c] / (rho_c - lam_{p+ua})
    tc_ok = tc_ok && cta_cgemm_tc(
        nu, p, n, [&](int ua, int r) { return c32(Z[(long long)r * nvec + p + ua], 0.f); },
        [&](int r, int c) { return C[(long long)r * p + c]; },
        [&](int ua, int c, c32 v) {
          coef[(long long)ua * p + c] = float(1.0 / (rho[c] - double(lam[p + ua]))) * v;
        },
        work, ts);
    __syncthreads();
    // update = Q_h D Z_u coef
    tc_ok = tc_ok && cta_cgemm_tc(
        n, p, nu, [&](int r, int ua) { return c32(Z[(long long)r * nvec + p + ua], 0.f); },
        [&](int ua, int c) { return coef[(long long)ua * p + c]; },
        [&](int r, int c, c32 v) { C[(long long)r * p + c] = Dp[r] * v; }, work, ts);
    __syncthreads();
    tc_ok = tc_ok && cta_reflect_wy(A, n, C, p, p, true, work, ts);
    // E = Q^dag Q - I with Q = Q32 + C: Q32^dag Q32 - I compensated (the FP32 basis is
    // orthonormal to ~1e-7, so the difference needs the extra precision), then the
    // small terms Q32^dag C + C^dag Q32 + C^dag C = D + D^dag, D = (Q32 + C / 2)^dag C, in FP32
    cta_gemm<GemmGramComp, false, true, CG_TILE, true>(
        p, p, n, [&](int x, int r) { return X[(long long)r * nbt + x]; },
        [&](int r, int y) { return X[(long long)r * nbt + y]; },
        [&](int x, int y, const CDF& acc) {
          z64 v = acc.value();
          if (x == y) v = z64(v.re - 1.0, 0.0);
          E[(long long)x * p + y] = c32(float(v.re), float(v.im));
          E[(long long)y * p + x] = c32(float(v.re), float(-v.im));
        },
        work);
    c32* F = E + (long long)p * p;
    __syncthreads();
    tc_ok = tc_ok && cta_cgemm_tc(
        p, p, n,
        [&](int x, int r) { return conj(X[(long long)r * nbt + x] + 0.5f * C[(long long)r * p + x]); },
        [&](int r, int y) { return C[(long long)r * p + y]; },
        [&](int x, int y, c32 v) { F[(long long)x * p + y] = v; }, work, ts);
    __syncthreads();
    for (int x = warp; x < p; x += nwarp)
      for (int y = lane; y < p; y += 32)
        E[(long long)x * p + y] = E[(long long)x * p + y] + F[(long long)x * p + y] + conj(F[(long long)y * p + x]);
    __syncthreads();
    // second order of (I + E)^{-1/2}: F = E - 3/4 E^2 (E reaches ~3e-5 where inverse iteration
    // leaves neighbouring vectors short of orthogonal, and E^2 would stay as the error)
    tc_ok = tc_ok && cta_cgemm_tc(
        p, p, p, [&](int x, int q) { return E[(long long)x * p + q]; },
        [&](int q, int y) { return E[(long long)q * p + y]; },
        [&](int x, int y, c32 v) { F[(long long)x * p + y] = E[(long long)x * p + y] - 0.75f * v; }, work, ts);
    __syncthreads();
    // Q = (Q32 + C) - (Q32 + C) F / 2, the correction in FP32
    tc_ok = tc_ok && cta_cgemm_tc(
        n, p, p, [&](int r, int q) { return X[(long long)r * nbt + q] + C[(long long)r * p + q]; },
        [&](int q, int c) { return F[(long long)q * p + c]; },
        [&](int r, int c, c32 v) {
          const c32 x32 = X[(long long)r * nbt + c], dc = C[(long long)r * p + c];
          Q[(long long)r * p + c] = z64(double(x32.re) + double(dc.re) - 0.5 * double(v.re),
                                        double(x32.im) + double(dc.im) - 0.5 * double(v.im));
        },
        work, ts);
    __syncthreads();
    if (!tc_ok && tid == 0) report(a.status, ST_ETIMEOUT, k, 0.0);
    // gap from FP64 Rayleigh quotients of the FP32 vectors p-1 and p: rho[p-1] is
    // already q^dag H q of vector p-1; H x_p by one warp per row (lanes along the row,
    // coalesced), in FP64
    if (a.polish) {
      // the polish takes the gap
    } else if (p < n) {
      double num = 0.0, den = 0.0, den1 = 0.0;
      for (int r = warp; r < n; r += nwarp) {
        z64 hv(0.0, 0.0);
        const int q0 = dense ? r * n : a.row_ptr[r], q1 = dense ? (r + 1) * n : a.row_ptr[r + 1];
        for (int q = q0 + lane; q < q1; q += 32) {
          const c32* hp = reinterpret_cast<const c32*>(He + q);
          const z64 h(double(hp[0].re) + double(hp[1].re), double(hp[0].im) + double(hp[1].im));
          cfma(hv, h, ccast<double>(X[(long long)(dense ? q - q0 : md.ent_col[q]) * nbt + p]));
        }
        for (int o = 16; o > 0; o >>= 1) {
          hv.re += __shfl_xor_sync(0xffffffffu, hv.re, o);
          hv.im += __shfl_xor_sync(0xffffffffu, hv.im, o);
        }
        if (lane == 0) {
          const z64 v = ccast<double>(X[(long long)r * nbt + p]);
          num += v.re * hv.re + v.im * hv.im;
          den += abs2(v);
          den1 += abs2(ccast<double>(X[(long long)r * nbt + p - 1]));
        }
      }
      num = block_sum(num, red);
      den = block_sum(den, red);
      den1 = block_sum(den1, red);
      if (tid == 0) {
        const double g = num / den - rho[p - 1] / den1;
        a.gap[k] = g;
        if (!(g > a.gap_tol)) report(a.status, ST_EGAP, k, g);
      }
    } else if (tid == 0) {
      a.gap[k] = INFINITY;
    }
    __syncthreads();
  }
  tc::teardown(ts);
}

// ---------------------------------------------------------------------------
// Stage 7 (FP64 request from the FP32 solve): one more Newton correction of the refined
// block Q, now to FP64 accuracy.
//   R = H Q - Q G, G = Q^dag H Q, and the Gram matrix in FP64; the complement's coefficients
//   and the correction C = Q_h D Z_u [Z_u^T D^dag Q_h^dag R / (rho - lam)] in FP32 (C is the
//   error that the first correction left, ~1e-12: FP32 keeps it to 1e-19); Q <- Q + C, then
//   Q <- Q - Q E / 2.
// The band edges: the largest eigenvalue of G, whose off-diagonal part is ~1e-6 ||H||, by
// three diagonally preconditioned corrections of its edge vectors (each takes a factor
// 1e-3 or more from their error) and their Ritz values; the smallest of the complement from
// the FP32 vectors of the upper edge, corrected like Q but against every level outside
// their cluster, made orthogonal to Q, by their Ritz values (error of the vectors
// (1e-6 ||H|| / width)^2, of the values its square).
// A k-point is left to the FP64 solve (need = 1) where this is not enough: a gap or an
// isolation of the edge clusters below 1e-3 of the spectral radius, told after the bisection
// (k_lg_polish_need), or |C| above 3e-9 here.  The FP32 basis is not renewed, so that |C| times
// its error e0 stays: at that bound 2e-16 ||H|| / gap for e0 ~ 6e-8 ||H|| / gap, the forward
// error of an FP64 solve.  H is scaled by a power of two, its unit does not matter.
//
// FP64 products bound it: four n p^2 (three of them on a sparse H) of the ~16/3 n^3 + 4 n^2 p
// that the FP64 tridiagonal solve takes, as tiled GEMMs instead of matrix-vector products.
// ---------------------------------------------------------------------------
__device__ __forceinline__ z64 block_csum(z64 v, double* red) {
  const double re = block_sum(v.re, red);
  return z64(re, block_sum(v.im, red));
}

// Y (n x g, leading dimension POLISH_G) = H X for a few columns (X, Y row-major), one warp
// per row.
template <class LX>
__device__ void polish_apply(const LargeArgs& a, const z64* He, int n, int g, LX x, z64* Y) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  for (int r = warp; r < n; r += nwarp) {
    const int q0 = a.row_ptr[r], q1 = a.row_ptr[r + 1];
    for (int b = 0; b < g; ++b) {
      z64 acc(0.0, 0.0);
      for (int q = q0 + lane; q < q1; q += 32) cfma(acc, He[q], x(a.model.ent_col[q], b));
      acc = warp_csum(acc);
      if (lane == 0) Y[r * POLISH_G + b] = acc;
    }
  }
}

// Orthonormal columns: modified Gram-Schmidt, twice, on g columns of length m.
__device__ void polish_mgs(z64* X, int m, int g, double* red) {
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int b = 0; b < g; ++b)
    for (int pass = 0; pass < 2; ++pass) {
      for (int q = 0; q < b; ++q) {
        z64 d(0.0, 0.0);
        for (int r = tid; r < m; r += nt) cfma_conj(d, X[r * POLISH_G + q], X[r * POLISH_G + b]);
        d = block_csum(d, red);
        for (int r = tid; r < m; r += nt) cfms(X[r * POLISH_G + b], X[r * POLISH_G + q], d);
      }
      double s = 0.0;
      for (int r = tid; r < m; r += nt) s += abs2(X[r * POLISH_G + b]);
      s = 1.0 / sqrt(block_sum(s, red));
      for (int r = tid; r < m; r += nt) X[r * POLISH_G + b] = s * X[r * POLISH_G + b];
      __syncthreads();
    }
}

// Extreme Ritz value of orthonormal columns X (m x g) with Y = (operator) X; E (g x g,
// leading dimension lde, <= 1e-8) the deviation of the metric from I, S - (E S + S E) / 2.
__device__ double polish_ritz(const z64* X, const z64* Y, int m, int g, bool want_max, const c32* E, int lde, z64* S,
                              z64* V, JacRot<double>* rot, double* red) {
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int x = 0; x < g; ++x)
    for (int y = x; y < g; ++y) {
      z64 d(0.0, 0.0);
      for (int r = tid; r < m; r += nt) cfma_conj(d, X[r * POLISH_G + x], Y[r * POLISH_G + y]);
      d = block_csum(d, red);
      if (tid == 0) {
        S[x * g + y] = x == y ? z64(d.re, 0.0) : d;
        if (x != y) S[y * g + x] = conj(d);
      }
    }
  __syncthreads();
  if (E) {
    z64 d(0.0, 0.0);
    const int x = tid / g, y = tid - x * g;
    if (x < g)
      for (int q = 0; q < g; ++q) {
        cfma(d, ccast<double>(E[x * lde + q]), S[q * g + y]);
        cfma(d, S[x * g + q], ccast<double>(E[q * lde + y]));
      }
    __syncthreads();
    if (x < g) S[x * g + y] = z64(S[x * g + y].re - 0.5 * d.re, x == y ? 0.0 : S[x * g + y].im - 0.5 * d.im);
    __syncthreads();
  }
  if (g > 1) jacobi_eigh<double>(S, V, g, g, 60, rot, red);
  double e = S[0].re;
  for (int c = 1; c < g; ++c) e = want_max ? fmax(e, S[c * g + c].re) : fmin(e, S[c * g + c].re);
  __syncthreads();
  return e;
}

template <int TN>
__global__ void __launch_bounds__(256, 2) k_lg_polish(LargeArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int n = a.n, p = a.p, nbt = a.nbt, nvec = a.nvec, tid = threadIdx.x, nt = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nwarp = nt >> 5;
  const DevModel& md = a.model;
  __shared__ double red[64];
  __shared__ z64 S[POLISH_G * POLISH_G], V[POLISH_G * POLISH_G];
  __shared__ JacRot<double> rot[POLISH_G];
  __shared__ double rhox[POLISH_G];
  __shared__ uint32_t tmem_slot;
  __shared__ __align__(8) uint64_t tc_bar;
  tc::State ts = tc::setup(&tmem_slot, &tc_bar);
  const int ldr = p + 4 * POLISH_G, ldc = p + POLISH_G;
  for (long long kw = blockIdx.x; kw < a.W; kw += gridDim.x) {
    const long long k = a.k0 + kw * (a.kstride > 0 ? a.kstride : 1);
    const c32* A = reinterpret_cast<const c32*>(a.A) + kw * (long long)n * n;
    const c32* Dp = reinterpret_cast<const c32*>(a.Dp) + kw * n;
    const float* Z = reinterpret_cast<const float*>(a.Z) + kw * (long long)nvec * n;
    const float* lam = reinterpret_cast<const float*>(a.lam) + kw * a.nval;
    const c32* X = reinterpret_cast<const c32*>(a.X) + kw * (long long)n * nbt;
    const z64* He = a.H64 + kw * (long long)md.n_ent;
    z64* Q = a.U + kw * (long long)n * p;
    z64* R = a.R64 + kw * (long long)n * ldr;          // H Q, later small blocks
    c32* C = a.C32 + kw * (long long)n * ldc;          // corrections: occupied, then upper edge
    z64* G = a.G64 + kw * ((long long)p * p + ((long long)p * p + 1) / 2);  // Q^dag H Q
    c32* E = reinterpret_cast<c32*>(G + (long long)p * p);  // Q^dag Q - I
    if (a.need[kw]) continue;  // uniform over the CTA
    const float width = polish_width(lam, n);
    const int g = polish_upper(lam, n, p), gl = polish_lower(lam, n, p);
    // R = H Q
    if (md.n_ent == n * n) {
      cta_gemm<GemmPlainT<double>, true, true, TN>(
          n, p, n, [&](int r, int q) { return He[(long long)r * n + q]; },
          [&](int q, int c) { return Q[(long long)q * p + c]; },
          [&](int r, int c, const z64& v) { R[(long long)r * ldr + c] = v; }, smem);
    } else {
      for (int r = warp; r < n; r += nwarp) {
        const int q0 = a.row_ptr[r], q1 = a.row_ptr[r + 1];
        for (int c = lane; c < p; c += 32) {
          z64 acc(0.0, 0.0);
          for (int q = q0; q < q1; ++q) cfma(acc, He[q], Q[(long long)md.ent_col[q] * p + c]);
          R[(long long)r * ldr + c] = acc;
        }
      }
    }
    __syncthreads();
    cta_gemm<GemmPlainT<double>, false, true, TN, true>(
        p, p, n, [&](int x, int r) { return conj(Q[(long long)r * p + x]); },
        [&](int r, int y) { return R[(long long)r * ldr + y]; },
        [&](int x, int y, const z64& v) {
          G[(long long)x * p + y] = x == y ? z64(v.re, 0.0) : v;
          if (x != y) G[(long long)y * p + x] = conj(v);
        },
        smem);
    __syncthreads();
    cta_gemm<GemmPlainT<double>, true, true, TN>(
        n, p, p, [&](int r, int q) { return Q[(long long)r * p + q]; },
        [&](int q, int c) { return G[(long long)q * p + c]; },
        [&](int r, int c, const z64& v) { C[(long long)r * ldc + c] = ccast<float>(R[(long long)r * ldr + c] - v); },
        smem);
    __syncthreads();
    // residuals of the upper edge's FP32 vectors x_b
    z64* XU = R;                            // n x POLISH_G blocks in the R workspace
    z64* YU = XU + (long long)n * POLISH_G;
    z64* XL = YU + (long long)n * POLISH_G; // p x POLISH_G
    z64* YL = XL + (long long)n * POLISH_G;
    polish_apply(a, He, n, g, [&](int q, int b) { return ccast<double>(X[(long long)q * nbt + p + b]); }, YU);
    __syncthreads();
    for (int b = 0; b < g; ++b) {
      double num = 0.0, den = 0.0;
      for (int r = tid; r < n; r += nt) {
        const z64 x = ccast<double>(X[(long long)r * nbt + p + b]), h = YU[r * POLISH_G + b];
        num += x.re * h.re + x.im * h.im;
        den += abs2(x);
      }
      num = block_sum(num, red);
      den = block_sum(den, red);
      const double rho = num / den;
      if (tid == 0) rhox[b] = rho;
      for (int r = tid; r < n; r += nt)
        C[(long long)r * ldc + p + b] =
            ccast<float>(YU[r * POLISH_G + b] - rho * ccast<double>(X[(long long)r * nbt + p + b]));
    }
    __syncthreads();
    // C <- D^dag Q_h^dag C
    bool tc_ok = cta_reflect_wy(A, n, C, p + g, ldc, false, smem, ts);
    for (int r = warp; r < n; r += nwarp) {
      const c32 d = conj(Dp[r]);
      for (int c = lane; c < p + g; c += 32) C[(long long)r * ldc + c] = d * C[(long long)r * ldc + c];
    }
    __syncthreads();
    // coefficients: occupied columns over the levels from p on, edge columns over every level
    // outside their cluster
    c32* coef = reinterpret_cast<c32*>(YL + (long long)n * POLISH_G);  // (n - p) x p, then n x POLISH_G
    c32* coefx = reinterpret_cast<c32*>(XL);
    const int nu = n - p;
    tc_ok = tc_ok && cta_cgemm_tc(
        nu, p, n, [&](int ua, int r) { return c32(Z[(long long)r * nvec + p + ua], 0.f); },
        [&](int r, int c) { return C[(long long)r * ldc + c]; },
        [&](int ua, int c, c32 v) {
          coef[(long long)ua * p + c] = float(1.0 / (G[(long long)c * p + c].re - double(lam[p + ua]))) * v;
        },
        smem, ts);
    for (int q = tid; q < n * g; q += nt) {
      const int b = q / n, l = q - b * n;
      c32 acc(0.f, 0.f);
      if (l < p || l >= p + g) {
        for (int r = 0; r < n; ++r) {
          const float z = Z[(long long)r * nvec + l];
          const c32 c = C[(long long)r * ldc + p + b];
          acc.re = fmaf(z, c.re, acc.re);
          acc.im = fmaf(z, c.im, acc.im);
        }
        // (a level just outside the cluster may come close to a far member of it; the edge
        // itself is a width away)
        const double dl = rhox[b] - double(lam[l]);
        acc = fabs(dl) > 0.1 * double(width) ? float(1.0 / dl) * acc : c32(0.f, 0.f);
      }
      coefx[l * POLISH_G + b] = acc;
    }
    __syncthreads();
    // C = Q_h D Z coef
    tc_ok = tc_ok && cta_cgemm_tc(
        n, p, nu, [&](int r, int ua) { return c32(Z[(long long)r * nvec + p + ua], 0.f); },
        [&](int ua, int c) { return coef[(long long)ua * p + c]; },
        [&](int r, int c, c32 v) { C[(long long)r * ldc + c] = Dp[r] * v; }, smem, ts);
    for (int r = warp; r < n; r += nwarp)
      for (int b = 0; b < g; ++b) {
        c32 acc(0.f, 0.f);
        for (int l = lane; l < n; l += 32) {
          const float z = Z[(long long)r * nvec + l];
          const c32 c = coefx[l * POLISH_G + b];
          acc.re = fmaf(z, c.re, acc.re);
          acc.im = fmaf(z, c.im, acc.im);
        }
        acc = warp_csum(acc);
        if (lane == 0) C[(long long)r * ldc + p + b] = Dp[r] * acc;
      }
    __syncthreads();
    tc_ok = tc_ok && cta_reflect_wy(A, n, C, p + g, ldc, true, smem, ts);
    __syncthreads();
    // Q <- Q + C; |C|^2
    double c2 = 0.0;
    for (int r = warp; r < n; r += nwarp)
      for (int c = lane; c < p; c += 32) {
        const c32 d = C[(long long)r * ldc + c];
        z64& q = Q[(long long)r * p + c];
        q = z64(q.re + double(d.re), q.im + double(d.im));
        c2 += double(abs2(d));
      }
    c2 = block_sum(c2, red);
    // E = Q^dag Q - I
    double emax = 0.0;
    cta_gemm<GemmPlainT<double>, false, true, TN, true>(
        p, p, n, [&](int x, int r) { return conj(Q[(long long)r * p + x]); },
        [&](int r, int y) { return Q[(long long)r * p + y]; },
        [&](int x, int y, const z64& v) {
          const c32 e(float(v.re - (x == y ? 1.0 : 0.0)), x == y ? 0.f : float(v.im));
          emax = fmax(emax, double(abs2(e)));
          E[(long long)x * p + y] = e;
          E[(long long)y * p + x] = conj(e);
        },
        smem);
    emax = -block_min(-emax, red);
    tc_ok = tc_ok && cta_cgemm_tc(
        n, p, p, [&](int r, int q) { return ccast<float>(Q[(long long)r * p + q]); },
        [&](int q, int c) { return E[(long long)q * p + c]; },
        [&](int r, int c, c32 v) { C[(long long)r * ldc + c] = v; }, smem, ts);
    __syncthreads();
    for (int r = warp; r < n; r += nwarp)
      for (int c = lane; c < p; c += 32) {
        const c32 d = C[(long long)r * ldc + c];
        z64& q = Q[(long long)r * p + c];
        q = z64(q.re - 0.5 * double(d.re), q.im - 0.5 * double(d.im));
      }
    if (!tc_ok && tid == 0) report(a.status, ST_ETIMEOUT, k, 0.0);
    if (!(c2 <= 1e-17) || !(emax <= 1e-16)) {  // uniform (block reductions)
      if (tid == 0) a.need[kw] = 1;
      __syncthreads();
      continue;
    }
    __syncthreads();
    // lower edge: vectors of G's last gl columns
    for (int e = tid; e < p * gl; e += nt) {
      const int r = e / gl, b = e - r * gl;
      XL[r * POLISH_G + b] = z64(double(r == p - gl + b), 0.0);
    }
    __syncthreads();
    auto apply_g = [&]() {
      for (int r = warp; r < p; r += nwarp)
        for (int b = 0; b < gl; ++b) {
          z64 acc(0.0, 0.0);
          for (int q = lane; q < p; q += 32) cfma(acc, G[(long long)r * p + q], XL[q * POLISH_G + b]);
          acc = warp_csum(acc);
          if (lane == 0) YL[r * POLISH_G + b] = acc;
        }
      __syncthreads();
    };
    for (int it = 0; it < 3; ++it) {
      apply_g();
      for (int e = tid; e < p * gl; e += nt) {
        const int r = e / gl, b = e - r * gl;
        const double rho = G[(long long)(p - gl + b) * p + p - gl + b].re;
        if (r < p - gl) {
          const double dl = rho - G[(long long)r * p + r].re;
          const double w = fabs(dl) > 0.1 * double(width) ? 1.0 / dl : 0.0;
          const z64 res = YL[r * POLISH_G + b] - rho * XL[r * POLISH_G + b];
          XL[r * POLISH_G + b] = XL[r * POLISH_G + b] + w * res;
        }
      }
      __syncthreads();
    }
    polish_mgs(XL, p, gl, red);
    apply_g();
    // (the columns that G was formed with were orthonormal to E)
    const double top = polish_ritz(XL, YL, p, gl, true, E + (long long)(p - gl) * p + p - gl, p, S, V, rot, red);
    // upper edge: the corrected vectors, orthogonal to Q
    for (int e = tid; e < n * g; e += nt) {
      const int r = e / g, b = e - r * g;
      const c32 x = X[(long long)r * nbt + p + b], c = C[(long long)r * ldc + p + b];
      XU[r * POLISH_G + b] = z64(double(x.re) + double(c.re), double(x.im) + double(c.im));
    }
    __syncthreads();
    for (int c = warp; c < p; c += nwarp)  // overlaps Q^dag x in XL
      for (int b = 0; b < g; ++b) {
        z64 acc(0.0, 0.0);
        for (int r = lane; r < n; r += 32) cfma_conj(acc, Q[(long long)r * p + c], XU[r * POLISH_G + b]);
        acc = warp_csum(acc);
        if (lane == 0) XL[c * POLISH_G + b] = acc;
      }
    __syncthreads();
    for (int r = warp; r < n; r += nwarp)
      for (int b = 0; b < g; ++b) {
        z64 acc(0.0, 0.0);
        for (int c = lane; c < p; c += 32) cfma(acc, Q[(long long)r * p + c], XL[c * POLISH_G + b]);
        acc = warp_csum(acc);
        if (lane == 0) XU[r * POLISH_G + b] = XU[r * POLISH_G + b] - acc;
      }
    __syncthreads();
    polish_mgs(XU, n, g, red);
    polish_apply(a, He, n, g, [&](int q, int b) { return XU[q * POLISH_G + b]; }, YU);
    __syncthreads();
    const double bot = polish_ritz(XU, YU, n, g, false, static_cast<c32*>(nullptr), 0, S, V, rot, red);
    if (tid == 0) {
      const double gp = (bot - top) / a.scale;
      a.gap[k] = gp;
      if (!(gp > a.gap_tol)) report(a.status, ST_EGAP, k, gp);
    }
    __syncthreads();
  }
  tc::teardown(ts);
}

// ---------------------------------------------------------------------------
// Launcher: every stage of one wave, in stream order.
// ---------------------------------------------------------------------------
namespace {
constexpr int LG_THREADS = 256;

int lg_grid(long long units) {
  const long long cap = 152LL * 4;
  return int(units < cap ? (units > 0 ? units : 1) : cap);
}

void lg_mark(const LargeArgs& a, const char* name) {
  if (a.mark) a.mark(a.mark_user, name);
}

template <typename T>
cudaError_t lg_common(const LargeArgs& a, cudaStream_t s) {
  k_lg_build<T><<<lg_grid(a.W), LG_THREADS, 0, s>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  lg_mark(a, "lg_build");
  // lower-triangle kernel: 5 n + (warps) n complex values of shared memory, with up
  // to 16 warps and at least 4; one CTA per SM keeps the matrices being reduced
  // resident in L2 (n = 256: 152 x 512 KB in complex64)
  const size_t vec_b = size_t(a.n) * sizeof(cx<T>), lim = size_t(200) << 10;
  const size_t fixed = 5 * vec_b + 64 * sizeof(double);
  // Each step waits on a few dependent L2 round trips, so several k-points per SM
  // (more CTAs with fewer warps each) hide more latency than more warps on one
  // k-point; a small wave gives each of its CTAs more warps instead.
  const int fit = fixed < lim ? int(std::min<size_t>(16, (lim - fixed) / vec_b)) : 0;
  const int want = a.W >= 4 * 152 ? 4 : (a.W >= 2 * 152 ? 8 : 16);
  const int warps = std::min(fit, want);
  // The matrix in shared memory where two CTAs of 8 warps or more fit an SM with it: every
  // column then sweeps it at shared-memory instead of L2 rates (with the five-barrier step:
  // n = 124, 256 k-points 4.9 -> 2.9 ms with the FP64 spin eigensolves; n = 127, 289 k-points
  // 1.12 -> 0.63).  One CTA per SM
  // with most of a larger matrix was slower than four on L2 (n = 256, 837 k-points: 11.2 ->
  // 14.0 ms): each step is a dozen dependent barriers that only other CTAs can hide.
  const size_t sm_s = fixed + 8 * vec_b + size_t(a.n) * (a.n + 1) / 2 * sizeof(cx<T>);
  static size_t cached_h = 0, cached_s = 0;
  if (sm_s + 1024 <= (size_t(227) << 10) / 2) {
    if ((e = set_smem_once(k_lg_tridiag_h<T, true>, sm_s, cached_s)) != cudaSuccess) return e;
    const long long per_sm = std::min<long long>(4, (227 << 10) / (long long)(sm_s + 1024));
    k_lg_tridiag_h<T, true><<<int(std::min<long long>(a.W, 152LL * per_sm)), 256, sm_s, s>>>(a);
  } else if (warps >= 4) {
    const size_t sm_h = fixed + size_t(warps) * vec_b;
    if ((e = set_smem_once(k_lg_tridiag_h<T, false>, sm_h, cached_h)) != cudaSuccess) return e;
    const long long ctas = std::min<long long>(a.W, 152LL * (16 / warps));
    k_lg_tridiag_h<T, false><<<int(ctas), 32 * warps, sm_h, s>>>(a);
  } else {
    const size_t sm_tri = 3 * size_t(a.n) * sizeof(cx<T>) + 64 * sizeof(double);
    static size_t cached = 0;
    if ((e = set_smem_once(k_lg_tridiag<T>, sm_tri, cached)) != cudaSuccess) return e;
    k_lg_tridiag<T><<<lg_grid(a.W), LG_THREADS, sm_tri, s>>>(a);
  }
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  lg_mark(a, "lg_tridiag");
  const size_t sm_b = bisect_smem<T>(a.n);
  static size_t cached_b = 0;
  if ((e = set_smem_once(k_lg_bisect<T>, sm_b, cached_b)) != cudaSuccess) return e;
  k_lg_bisect<T><<<dim3(unsigned(std::min<long long>(a.W, 65535)), unsigned((a.nval + BIS_THREADS - 1) / BIS_THREADS)),
                   BIS_THREADS, sm_b, s>>>(a);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (sizeof(T) == 4 && a.polish) {
    k_lg_polish_need<<<1, 256, 0, s>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  lg_mark(a, "lg_bisect");
  const long long ni = a.W * a.nvec;
  if (ni > 0) {
    if (a.subspace_only) {
      k_lg_invit_par<T><<<int((ni + 63) / 64), 64, 0, s>>>(a);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      const long long nw = ni * 32;
      if (nw / 128 + 1 > 0x7fffffffLL) return cudaErrorInvalidValue;
      k_lg_invit_orth<T><<<int((nw + 127) / 128), 128, 0, s>>>(a);
    } else {
      k_lg_invit<T><<<int((ni + 63) / 64), 64, 0, s>>>(a);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    lg_mark(a, "lg_invit");
  }
  return cudaSuccess;
}
}  // namespace

cudaError_t launch_states_large(const LargeArgs& a, cudaStream_t s) {
  if (a.W <= 0) return cudaSuccess;
  cudaError_t e;
  if (!a.mixed) {
    if ((e = lg_common<double>(a, s)) != cudaSuccess) return e;
    if (a.p == 0) return cudaSuccess;  // values only
    // one-reflector panels while a panel holds at least 16 columns (n <= ~780); beyond,
    // a panel of a few columns would sweep every reflector once per few columns, so
    // the reflectors are applied in compact-WY blocks through FP64 GEMMs (pw = 0)
    const int pw = reflect_pw<double>(a.n, size_t(200) << 10);
    if (pw >= 16) {
      const size_t sm = reflect_smem<double>(a.n, pw);
      static size_t cached = 0;
      if ((e = set_smem_once(k_lg_backtransform<double, double>, sm, cached)) != cudaSuccess) return e;
      k_lg_backtransform<double, double><<<lg_grid(a.W), LG_THREADS, sm, s>>>(
          a, a.U, (long long)a.n * a.p, a.p, pw);
    } else {
      const size_t sm = reflect_wy_simt_smem<double>();
      static size_t cached_wy = 0;
      if ((e = set_smem_once(k_lg_backtransform_wy64, sm, cached_wy)) != cudaSuccess) return e;
      k_lg_backtransform_wy64<<<lg_grid(a.W), LG_THREADS, sm, s>>>(a, a.U, (long long)a.n * a.p, a.p);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    lg_mark(a, "lg_backtransform");
    if (a.Hin) return cudaSuccess;  // batched eigensolve: every eigenvalue is returned, no gap test
    k_lg_gap64<<<int((a.W + 127) / 128), 128, 0, s>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    lg_mark(a, "lg_gap");
    return cudaSuccess;
  }
  if ((e = lg_common<float>(a, s)) != cudaSuccess) return e;
  if (a.no_refine) return cudaSuccess;
  const size_t sm = reflect_wy_smem();
  static size_t cached = 0;
  if ((e = set_smem_once(k_lg_backtransform<float, float>, sm, cached)) != cudaSuccess) return e;
  k_lg_backtransform<float, float><<<lg_grid(a.W), LG_THREADS, sm, s>>>(
      a, reinterpret_cast<c32*>(a.X), (long long)a.n * a.nbt, a.nbt, 0);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  lg_mark(a, "lg_backtransform");
  const size_t smr = refine_work_offset(a.p) + std::max(std::max(reflect_wy_smem(), tc::SMEM), CG_SMEM);
  static size_t cached_r = 0;
  if ((e = set_smem_once(k_lg_refine, smr, cached_r)) != cudaSuccess) return e;
  k_lg_refine<<<lg_grid(a.W), LG_THREADS, smr, s>>>(a);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  lg_mark(a, "lg_refine");
  if (a.polish) {
    const size_t smp = std::max(std::max(reflect_wy_smem(), tc::SMEM), cg_smem<GemmPlainT<double>>());
    static size_t cached_p32 = 0, cached_p64 = 0;
    if (a.p <= 32) {
      if ((e = set_smem_once(k_lg_polish<32>, smp, cached_p32)) != cudaSuccess) return e;
      k_lg_polish<32><<<lg_grid(a.W), LG_THREADS, smp, s>>>(a);
    } else {
      if ((e = set_smem_once(k_lg_polish<64>, smp, cached_p64)) != cudaSuccess) return e;
      k_lg_polish<64><<<lg_grid(a.W), LG_THREADS, smp, s>>>(a);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    lg_mark(a, "lg_polish");
  }
  return cudaSuccess;
}

// ---------------------------------------------------------------------------
// Batched eigensolve of explicit matrices: FP64 Rayleigh-Ritz of the refined block
// (mixed path, p <= 64) and the scatter of eigenvalues / eigenvectors to the
// caller's packed layout.
// ---------------------------------------------------------------------------
__global__ void k_eigh_ritz(LargeArgs a, double* ritz) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int n = a.n, p = a.p, tid = threadIdx.x, nt = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nwarp = nt >> 5;
  z64* G = reinterpret_cast<z64*>(smem);    // p x p
  z64* V = G + p * p;                       // p x p
  JacRot<double>* rot = reinterpret_cast<JacRot<double>*>(V + p * p);
  double* red = reinterpret_cast<double*>(rot + (p / 2 + 2));
  int* ord = reinterpret_cast<int*>(red + 64);
  for (long long kw = blockIdx.x; kw < a.W; kw += gridDim.x) {
    const c32* He = reinterpret_cast<const c32*>(a.Hent + kw * (long long)n * n);
    z64* Q = a.U + kw * (long long)n * p;
    z64* HQ = a.R64 + kw * (long long)n * p;
    for (int r = warp; r < n; r += nwarp)  // H Q in FP64 (H from its float-pair split)
      for (int c = lane; c < p; c += 32) {
        z64 acc(0.0, 0.0);
        for (int q = 0; q < n; ++q) {
          const c32 hi = He[2 * ((long long)r * n + q)], lo = He[2 * ((long long)r * n + q) + 1];
          cfma(acc, z64(double(hi.re) + double(lo.re), double(hi.im) + double(lo.im)), Q[(long long)q * p + c]);
        }
        HQ[(long long)r * p + c] = acc;
      }
    __syncthreads();
    for (int e = tid; e < p * p; e += nt) {
      const int x = e / p, y = e - x * p;
      z64 acc(0.0, 0.0);
      for (int r = 0; r < n; ++r) cfma_conj(acc, Q[(long long)r * p + x], HQ[(long long)r * p + y]);
      G[e] = acc;
    }
    __syncthreads();
    for (int e = tid; e < p * p; e += nt) {  // Hermitian part
      const int x = e / p, y = e - x * p;
      if (x < y) {
        const z64 h = 0.5 * (G[x * p + y] + conj(G[y * p + x]));
        G[x * p + y] = h;
        G[y * p + x] = conj(h);
      } else if (x == y) {
        G[e] = z64(G[e].re, 0.0);
      }
    }
    __syncthreads();
    const int sw = jacobi_eigh<double>(G, V, p, p, 40, rot, red);
    if (sw < 0 && tid == 0) report(a.status, ST_ENOCONV, a.k0 + kw, 0.0);
    sort_diag(G, p, p, ord);
    for (int c = tid; c < p; c += nt) ritz[kw * p + c] = G[ord[c] * p + ord[c]].re;
    // Q <- Q V (columns in ascending order), row by row through HQ as scratch
    for (int r = warp; r < n; r += nwarp)
      for (int c = lane; c < p; c += 32) {
        z64 acc(0.0, 0.0);
        for (int q = 0; q < p; ++q) cfma(acc, Q[(long long)r * p + q], V[q * p + ord[c]]);
        HQ[(long long)r * p + c] = acc;
      }
    __syncthreads();
    for (long long e = tid; e < (long long)n * p; e += nt) Q[e] = HQ[e];
    __syncthreads();
  }
}

cudaError_t launch_eigh_ritz(const LargeArgs& a, double* ritz, cudaStream_t s) {
  if (a.W <= 0 || a.p <= 0) return cudaSuccess;
  if (a.p > 64) return cudaErrorInvalidValue;
  const size_t sm = 2 * size_t(a.p) * a.p * sizeof(z64) + (a.p / 2 + 2) * sizeof(JacRot<double>) +
                    64 * sizeof(double) + size_t(a.p) * sizeof(int) + 16;
  static size_t cached = 0;
  cudaError_t e = set_smem_once(k_eigh_ritz, sm, cached);
  if (e != cudaSuccess) return e;
  k_eigh_ritz<<<lg_grid(a.W), LG_THREADS, sm, s>>>(a, ritz);
  return cudaGetLastError();
}

__global__ void k_eigh_scatter(EighScatterArgs e) {
  for (long long kw = blockIdx.x; kw < e.W; kw += gridDim.x) {
    const int b = e.idx[e.k0 + kw];
    double* ev = e.evals + e.e_off[b];
    for (int i = threadIdx.x; i < e.n; i += blockDim.x) {
      double v;
      if (e.ritz && i < e.p)
        v = e.ritz[kw * e.p + i];
      else if (e.mixed)
        v = double(reinterpret_cast<const float*>(e.lam)[kw * e.nval + i]);
      else
        v = reinterpret_cast<const double*>(e.lam)[kw * e.nval + i];
      ev[i] = v;
    }
    if (e.evecs && e.p > 0) {
      const z64* src = e.U + kw * (long long)e.n * e.p;
      z64* dst = e.evecs + e.v_off[b];
      for (long long x = threadIdx.x; x < (long long)e.n * e.p; x += blockDim.x) dst[x] = src[x];
    }
  }
}

cudaError_t launch_eigh_scatter(const EighScatterArgs& e, cudaStream_t s) {
  if (e.W <= 0) return cudaSuccess;
  k_eigh_scatter<<<lg_grid(e.W), 256, 0, s>>>(e);
  return cudaGetLastError();
}

}  // namespace bw
