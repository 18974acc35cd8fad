// Block-wide two-sided Jacobi eigensolver for a Hermitian matrix in shared memory.
//
// Parallel cyclic Jacobi with round-robin pairing: each round rotates n/2 disjoint
// index pairs at once, n-1 rounds make a sweep, and
// sweeps repeat until the off-diagonal Frobenius norm falls below 8 eps ||A||_F.
// A complex 2x2 rotation J = [[c, s e^{i phi}], [-s e^{-i phi}, c]] annihilates
// A[p][q] = |b| e^{i phi}: with tau = (A_qq - A_pp) / (2|b|) and
// t = sign(tau) / (|tau| + sqrt(1 + tau^2)), c = 1/sqrt(1+t^2), s = t c, and
// A_pp -> A_pp - t|b|, A_qq -> A_qq + t|b|.  A rotation is skipped when
// |A_pq| <= 4 eps sqrt(|A_pp| |A_qq|) (negligible against its diagonal pair); a sweep
// without any rotation also ends the iteration.  Without that test, clusters of
// equal eigenvalues keep off-diagonal entries at the rounding level that no
// rotation removes, and a pure norm test may never be met in FP32.
#pragma once

#include "common.cuh"

namespace bw {

template <typename T>
struct JacRot {
  int p, q;
  T c, app, aqq;
  cx<T> sc;  // s e^{i phi}
};

template <typename T>
__device__ __forceinline__ T eps_of();
template <>
__device__ __forceinline__ double eps_of<double>() { return 2.220446049250313e-16; }
template <>
__device__ __forceinline__ float eps_of<float>() { return 1.1920929e-7f; }

// Round-robin pair k of round r over np (even) players; indices >= n are dummies.
__device__ __forceinline__ void rr_pair(int r, int k, int np, int& p, int& q) {
  const int m = np - 1;
  if (k == 0) {
    p = m;
    q = r;
  } else {
    p = (r + k) % m;
    q = (r - k + m) % m;
  }
  if (p > q) { int t = p; p = q; q = t; }
}

// Diagonalises A (n x n, leading dimension ld) in place and accumulates V = prod J.
// On return A's diagonal holds the eigenvalues (unsorted).  rot: >= n/2+1 JacRot
// slots; red: >= 32 doubles.  Returns the number of sweeps, or -1 without
// convergence after max_sweeps.  turned (shared memory, optional) receives the number of
// rotations.  Every thread of the block must call it.
template <typename T>
__device__ int jacobi_eigh(cx<T>* A, cx<T>* V, int n, int ld, int max_sweeps, JacRot<T>* rot,
                           double* red, int* turned = nullptr) {
  const int tid = threadIdx.x, nt = blockDim.x;
  int count = 0;
  auto done = [&](int result) {
    if (turned) {
      const double all = block_sum(double(count), red);
      if (tid == 0) *turned = int(all);
      __syncthreads();
    }
    return result;
  };
  for (int e = tid; e < n * n; e += nt) {
    const int r = e / n, c = e - r * n;
    V[r * ld + c] = cx<T>(T(r == c), T(0));
  }
  if (n == 1) {
    __syncthreads();
    return done(0);
  }
  const int np = (n + 1) & ~1, npairs = np >> 1;
  // ||A||_F (invariant under the rotations)
  double fro = 0.0;
  for (int e = tid; e < n * n; e += nt) {
    const int r = e / n, c = e - r * n;
    fro += double(abs2(A[r * ld + c]));
  }
  fro = block_sum(fro, red);
  const double tol = 8.0 * double(eps_of<T>()) * sqrt(fro);
  __shared__ int s_rotated;
  [[maybe_unused]] __shared__ int s_list[32], s_turns;  // FP64 only
  for (int sweep = 0; sweep <= max_sweeps; ++sweep) {
    double off = 0.0;
    for (int e = tid; e < n * n; e += nt) {
      const int r = e / n, c = e - r * n;
      if (r != c) off += double(abs2(A[r * ld + c]));
    }
    off = block_sum(off, red);
    if (sqrt(off) <= tol || fro == 0.0) return done(sweep);
    if (sweep == max_sweeps) break;
    if (tid == 0) s_rotated = 0;
    __syncthreads();
    for (int r = 0; r < np - 1; ++r) {
      for (int k = tid; k < npairs; k += nt) {
        int p, q;
        rr_pair(r, k, np, p, q);
        JacRot<T> R;
        R.p = p;
        R.q = q;
        R.c = T(1);
        R.sc = cx<T>(T(0), T(0));
        R.app = T(0);
        R.aqq = T(0);
        if (q < n) {
          const cx<T> b = A[p * ld + q];
          const T a = A[p * ld + p].re, d = A[q * ld + q].re;
          R.app = a;
          R.aqq = d;
          const T b2 = abs2(b), e4 = T(4) * eps_of<T>();
          if (b2 > e4 * e4 * fabs(a) * fabs(d) && b2 > T(0)) {
            s_rotated = 1;
            ++count;
            T ab, t, c, s;  // s = sin / |b|
            if constexpr (sizeof(T) == 4) {
              // hardware reciprocal roots with a Newton step for what keeps the rotation
              // unitary (c and 1 / |b|); the angle itself may be off by an ulp or two
              auto inv_root = [](float x) {
                const float y = rsqrtf(x);
                return fmaf(0.5f * y, fmaf(-x * y, y, 1.f), y);
              };
              const float iab = inv_root(b2), tau = 0.5f * (d - a) * iab;
              ab = b2 * iab;
              t = copysignf(__frcp_rn(fabsf(tau) + sqrtf(fmaf(tau, tau, 1.f))), tau >= 0.f ? 1.f : -1.f);
              c = inv_root(fmaf(t, t, 1.f));
              s = t * c * iab;
            } else {
              ab = sqrt(b2);
              const T tau = (d - a) / (T(2) * ab);
              t = (tau >= T(0) ? T(1) : T(-1)) / (fabs(tau) + sqrt(T(1) + tau * tau));
              c = T(1) / sqrt(T(1) + t * t);
              s = t * c / ab;
            }
            R.c = c;
            R.sc = cx<T>(s * b.re, s * b.im);
            R.app = a - t * ab;
            R.aqq = d + t * ab;
          }
        } else {
          R.q = -1;  // dummy pair
        }
        rot[k] = R;
      }
      if constexpr (sizeof(T) == 8) {
        // the pairs that turn, then the others (n <= 64: one warp holds them all)
        if (tid < 32) {
          const bool turns = tid < npairs && rot[tid].q >= 0 && (rot[tid].sc.re != T(0) || rot[tid].sc.im != T(0));
          const unsigned mask = __ballot_sync(0xffffffffu, turns), before = mask & ((1u << tid) - 1u);
          if (tid < npairs) s_list[turns ? __popc(before) : __popc(mask) + tid - __popc(before)] = tid;
          if (tid == 0) s_turns = __popc(mask);
        }
      }
      __syncthreads();
      // A <- J^dagger A J by 2 x 2 blocks (pair k1's rows, pair k2's columns) and V <- V J by
      // pairs and rows, in one phase: two barriers per round (four, with the rows and the
      // columns apart, held n = 32 to 15 % issue).  Consecutive threads take consecutive pairs
      // of a row, so their accesses spread over the banks.  Spin-resolved n = 32, 441 k-points:
      // states 1.65 -> 0.90 ms; n = 24, 961 k-points 1.22 -> 0.90 ms.
      if constexpr (sizeof(T) == 8) {
        // FP64 operations bound it, so only the pairs that turn are worked on: blocks of their
        // rows (e < nr), of their columns in the other rows (e < nr + nc), columns of V, the
        // threads of a warp alike.  Late sweeps, and matrices that keep most entries at zero, turn
        // few pairs of a round: eight random blocks, n = 32, 3721 k-points 17.1 -> 6.3 ms, dense
        // matrices of n = 32 33.4 -> 29.4 ms.
        const int m = s_turns, nr = m * npairs, nc = m * (npairs - m);
        if (npairs <= 4) {
          // one warp: rows, then columns, two outputs to a thread each (sixteen blocks of eight
          // leave half of it idle: n = 8, 3721 matrices 1.25 -> 0.98 ms)
          for (int e = tid; e < m * n; e += nt) {
            const int col = e / m;
            const JacRot<T> P = rot[s_list[e - col * m]];
            const cx<T> ap = A[P.p * ld + col], aq = A[P.q * ld + col];
            A[P.p * ld + col] = P.c * ap - P.sc * aq;
            A[P.q * ld + col] = conj(P.sc) * ap + P.c * aq;
          }
          __syncthreads();
          for (int e = tid; e < m * n; e += nt) {
            const int row = e / m;
            const JacRot<T> Q = rot[s_list[e - row * m]];
            cx<T>* ra = A + row * ld;
            const cx<T> ap = ra[Q.p], aq = ra[Q.q];
            const bool pp = row == Q.p, qq = row == Q.q;  // the annihilated pair and its diagonal
            ra[Q.p] = pp ? cx<T>(Q.app, T(0)) : qq ? cx<T>(T(0), T(0)) : Q.c * ap - aq * conj(Q.sc);
            ra[Q.q] = qq ? cx<T>(Q.aqq, T(0)) : pp ? cx<T>(T(0), T(0)) : ap * Q.sc + Q.c * aq;
            const cx<T> vp = V[row * ld + Q.p], vq = V[row * ld + Q.q];
            V[row * ld + Q.p] = Q.c * vp - vq * conj(Q.sc);
            V[row * ld + Q.q] = vp * Q.sc + Q.c * vq;
          }
          __syncthreads();
          continue;
        }
        for (int e = tid; e < nr + nc + m * n; e += nt) {
          if (e >= nr + nc) {
            const int row = (e - nr - nc) / m;
            const JacRot<T> Q = rot[s_list[e - nr - nc - row * m]];
            const cx<T> vp = V[row * ld + Q.p], vq = V[row * ld + Q.q];
            V[row * ld + Q.p] = Q.c * vp - vq * conj(Q.sc);
            V[row * ld + Q.q] = vp * Q.sc + Q.c * vq;
            continue;
          }
          const int i1 = e < nr ? e / npairs : (e - nr) / m;
          const int i2 = e < nr ? e - i1 * npairs : e - nr - i1 * m;
          const JacRot<T> P = rot[s_list[e < nr ? i1 : m + i1]], Q = rot[s_list[i2]];
          if (e < nr && i1 == i2) {  // the annihilated pair and its diagonal
            A[P.p * ld + P.q] = cx<T>(T(0), T(0));
            A[P.q * ld + P.p] = cx<T>(T(0), T(0));
            A[P.p * ld + P.p] = cx<T>(P.app, T(0));
            A[P.q * ld + P.q] = cx<T>(P.aqq, T(0));
            continue;
          }
          const bool q1 = P.q >= 0, q2 = Q.q >= 0;
          const cx<T> zero(T(0), T(0));
          cx<T>* rp = A + P.p * ld;
          cx<T>* rq = A + (q1 ? P.q : P.p) * ld;
          cx<T> a00 = rp[Q.p], a01 = q2 ? rp[Q.q] : zero;
          cx<T> a10 = q1 ? rq[Q.p] : zero, a11 = q1 && q2 ? rq[Q.q] : zero;
          if (e < nr) {
            const cx<T> b00 = P.c * a00 - P.sc * a10, b01 = P.c * a01 - P.sc * a11;
            a10 = conj(P.sc) * a00 + P.c * a10;
            a11 = conj(P.sc) * a01 + P.c * a11;
            a00 = b00;
            a01 = b01;
          }
          if (i2 < m) {
            const cx<T> b00 = Q.c * a00 - a01 * conj(Q.sc), b10 = Q.c * a10 - a11 * conj(Q.sc);
            a01 = a00 * Q.sc + Q.c * a01;
            a11 = a10 * Q.sc + Q.c * a11;
            a00 = b00;
            a10 = b10;
          }
          rp[Q.p] = a00;
          if (q2) rp[Q.q] = a01;
          if (q1) rq[Q.p] = a10;
          if (q1 && q2) rq[Q.q] = a11;
        }
      } else {
        const int nblk = npairs * npairs;
        for (int e = tid; e < nblk + npairs * n; e += nt) {
          const int k1 = e < nblk ? e / npairs : (e - nblk) / npairs;
          const int k2 = e < nblk ? e - k1 * npairs : e - nblk - k1 * npairs;
          const JacRot<T> Q = rot[k2];
          const bool q2 = Q.q >= 0, id2 = Q.sc.re == T(0) && Q.sc.im == T(0);
          if (e >= nblk) {  // row k1 of V
            if (!q2 || id2) continue;
            const cx<T> vp = V[k1 * ld + Q.p], vq = V[k1 * ld + Q.q];
            V[k1 * ld + Q.p] = Q.c * vp - vq * conj(Q.sc);
            V[k1 * ld + Q.q] = vp * Q.sc + Q.c * vq;
            continue;
          }
          const JacRot<T> P = rot[k1];
          const bool q1 = P.q >= 0, id1 = P.sc.re == T(0) && P.sc.im == T(0);
          if (id1 && id2) continue;
          if (k1 == k2) {  // the annihilated pair and its diagonal
            A[P.p * ld + P.q] = cx<T>(T(0), T(0));
            A[P.q * ld + P.p] = cx<T>(T(0), T(0));
            A[P.p * ld + P.p] = cx<T>(P.app, T(0));
            A[P.q * ld + P.q] = cx<T>(P.aqq, T(0));
            continue;
          }
          const cx<T> zero(T(0), T(0));
          cx<T>* rp = A + P.p * ld;
          cx<T>* rq = A + (q1 ? P.q : P.p) * ld;
          const cx<T> a00 = rp[Q.p], a01 = q2 ? rp[Q.q] : zero;
          const cx<T> a10 = q1 ? rq[Q.p] : zero, a11 = q1 && q2 ? rq[Q.q] : zero;
          const cx<T> b00 = P.c * a00 - P.sc * a10, b01 = P.c * a01 - P.sc * a11;
          const cx<T> b10 = conj(P.sc) * a00 + P.c * a10, b11 = conj(P.sc) * a01 + P.c * a11;
          rp[Q.p] = Q.c * b00 - b01 * conj(Q.sc);
          if (q2) rp[Q.q] = b00 * Q.sc + Q.c * b01;
          if (q1) rq[Q.p] = Q.c * b10 - b11 * conj(Q.sc);
          if (q1 && q2) rq[Q.q] = b10 * Q.sc + Q.c * b11;
        }
      }
      __syncthreads();
    }
    if (!s_rotated) return done(sweep + 1);
  }
  return done(-1);
}

// Sort key that puts NaN after every number, so that ranks always form a
// permutation (NaN only appears when the input was not finite).
template <typename T>
__device__ __forceinline__ T rank_key(T x) { return isnan(x) ? T(INFINITY) : x; }

// order[rank] = index of the rank-th smallest diagonal entry (stable, NaN last).
template <typename T>
__device__ void sort_diag(const cx<T>* A, int n, int ld, int* order) {
  for (int a = threadIdx.x; a < n; a += blockDim.x) {
    const T la = rank_key(A[a * ld + a].re);
    int rank = 0;
    for (int b = 0; b < n; ++b) {
      const T lb = rank_key(A[b * ld + b].re);
      rank += (lb < la) || (lb == la && b < a);
    }
    order[rank] = a;
  }
  __syncthreads();
}

}  // namespace bw
