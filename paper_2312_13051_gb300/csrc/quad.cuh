// Four lanes per k-point for four-band models: lane l of a group of four
// consecutive lanes holds row l of H(k) and of the eigenvector matrix.  Shared by
// the states kernels (tiny.cu) and the fused mixed-precision loop kernel (loops.cu).
//
// A Jacobi sweep is three rounds; round R rotates the disjoint pairs {l, l ^ R} at
// once, the two lanes of a pair compute the same rotation, partner rows travel by
// warp shuffles, and every lane applies both rotations of the round to the columns
// of its own rows.  The mixed-precision solve (quad_df_occupied) runs the sweeps in
// FP32 on a double-float Hamiltonian and refines the occupied pair to double-float
// accuracy.
#pragma once

#include "common.cuh"
#include "df32.cuh"

namespace bw {

template <typename T>
__device__ __forceinline__ T teps();
template <>
__device__ __forceinline__ double teps<double>() { return 2.220446049250313e-16; }
template <>
__device__ __forceinline__ float teps<float>() { return 1.1920929e-7f; }

__device__ __forceinline__ int pmod(long long x, int m) {
  long long r = x % m;
  return int(r < 0 ? r + m : r);
}

struct TabShape {
  int B, H;  // low-level entries (w^0 .. w^{B-1}), high-level entries (w^{0}, w^{B}, ...)
};

template <typename T>
__device__ __forceinline__ cx<T> shfl_z(cx<T> v, int src) {
  return cx<T>(__shfl_sync(0xffffffffu, v.re, src), __shfl_sync(0xffffffffu, v.im, src));
}

// x[i] for a runtime i in [0, 4) without dynamic register indexing.
template <typename E>
__device__ __forceinline__ E sel4(const E (&x)[4], int i) {
  E r = x[0];
  if (i == 1) r = x[1];
  if (i == 2) r = x[2];
  if (i == 3) r = x[3];
  return r;
}

// Rotation of the Hermitian 2 x 2 block (a, b; conj b, d): c, s e^{i phi} and t as in
// the one-thread solver; false when the off-diagonal entry is negligible.
template <typename T>
__device__ __forceinline__ bool quad_angle(T a, T d, cx<T> b, T& c, cx<T>& sc, T& t, T& ab) {
  ab = sqrt(abs2(b));
  if (!(ab > T(4) * teps<T>() * sqrt(fabs(a) * fabs(d)) && ab > T(0))) return false;
  const T tau = (d - a) / (T(2) * ab);
  t = (tau >= T(0) ? T(1) : T(-1)) / (fabs(tau) + sqrt(T(1) + tau * tau));
  c = T(1) / sqrt(T(1) + t * t);
  const T s = t * c / ab;
  sc = cx<T>(s * b.re, s * b.im);
  return true;
}

// FP32 rotation from hardware reciprocal square roots and reciprocals (about 2 ulp):
// the FP32 sweeps only seed the double-float refinement, whose result does not
// depend on the last bits of the rotations.  The skip test compares squares.
template <>
__device__ __forceinline__ bool quad_angle<float>(float a, float d, c32 b, float& c, c32& sc, float& t,
                                                  float& ab) {
  const float b2 = abs2(b);
  const float e4 = 4.f * teps<float>();
  if (!(b2 > e4 * e4 * fabsf(a) * fabsf(d) && b2 > 0.f)) {
    ab = 0.f;
    return false;
  }
  const float inv_ab = rsqrtf(b2);
  ab = b2 * inv_ab;
  const float tau = 0.5f * (d - a) * inv_ab;
  t = copysignf(__frcp_rn(fabsf(tau) + sqrtf(fmaf(tau, tau, 1.f))), tau);
  if (tau == 0.f) t = 1.f;
  c = rsqrtf(fmaf(t, t, 1.f));
  const float s = t * c * inv_ab;
  sc = c32(s * b.re, s * b.im);
  return true;
}

template <int R, typename T>
__device__ __forceinline__ bool quad_round(cx<T> (&Ar)[4], cx<T> (&Vr)[4], int l, int base,
                                           bool frozen) {
  constexpr int Q = R == 1 ? 2 : 1;          // a lane of the other pair is l ^ Q
  constexpr int A0 = 0, A1 = R;              // pair containing index 0
  constexpr int B0 = R == 1 ? 2 : 1, B1 = R == 3 ? 2 : 3;  // the other pair
  const int partner = l ^ R;
  const bool is_p = l < partner;
  const T own_d = sel4(Ar, l).re;
  const T par_d = __shfl_sync(0xffffffffu, own_d, base + partner);
  const cx<T> bo = sel4(Ar, partner);
  const cx<T> b = is_p ? bo : conj(bo);      // A[p][q] from either row (exact Hermitian storage)
  const T a = is_p ? own_d : par_d, d = is_p ? par_d : own_d;
  T c = T(1), t = T(0), ab = T(0);
  cx<T> sc(T(0), T(0));
  const bool rot = !frozen && quad_angle(a, d, b, c, sc, t, ab);
  // rows: own row with the partner's
  cx<T> other[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) other[k] = shfl_z(Ar[k], base + partner);
  if (rot) {
    const cx<T> beta = is_p ? cx<T>(-sc.re, -sc.im) : conj(sc);
#pragma unroll
    for (int k = 0; k < 4; ++k) Ar[k] = c * Ar[k] + beta * other[k];
  }
  // columns: both rotations of the round on the own row of A and of V
  const T c2 = __shfl_sync(0xffffffffu, c, base + (l ^ Q));
  const cx<T> sc2 = shfl_z(sc, base + (l ^ Q));
  const bool mine_a = (l == A0 || l == A1);
  const T cA = mine_a ? c : c2, cB = mine_a ? c2 : c;
  const cx<T> sA = mine_a ? sc : sc2, sB = mine_a ? sc2 : sc;
  {
    const cx<T> ap = Ar[A0], aq = Ar[A1];
    Ar[A0] = cA * ap - aq * conj(sA);
    Ar[A1] = ap * sA + cA * aq;
    const cx<T> vp = Vr[A0], vq = Vr[A1];
    Vr[A0] = cA * vp - vq * conj(sA);
    Vr[A1] = vp * sA + cA * vq;
  }
  {
    const cx<T> ap = Ar[B0], aq = Ar[B1];
    Ar[B0] = cB * ap - aq * conj(sB);
    Ar[B1] = ap * sB + cB * aq;
    const cx<T> vp = Vr[B0], vq = Vr[B1];
    Vr[B0] = cB * vp - vq * conj(sB);
    Vr[B1] = vp * sB + cB * vq;
  }
  if (rot) {  // the annihilated entry and the new diagonal, as in the one-thread solver
    const cx<T> dnew(is_p ? a - t * ab : d + t * ab, T(0));
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (k == partner) Ar[k] = cx<T>(T(0), T(0));
      if (k == l) Ar[k] = dnew;
    }
  }
  return rot;
}

// Parallel-ordered Jacobi on the group's 4 x 4 matrix (lane l holds row l of A and
// of V, V starting as the identity).  Returns the sweeps used, or -1 without
// convergence within max_sweeps.  The warp's groups sweep together (the rounds
// shuffle across the whole warp): a converged group is frozen, its rotations the
// identity, until every group of the warp has converged.
template <typename T>
__device__ __forceinline__ int quad_jacobi(cx<T> (&Ar)[4], cx<T> (&Vr)[4], int l, int base,
                                           int max_sweeps) {
#pragma unroll
  for (int c = 0; c < 4; ++c) Vr[c] = cx<T>(T(c == l), T(0));
  T fro = T(0);
#pragma unroll
  for (int c = 0; c < 4; ++c) fro += abs2(Ar[c]);
  fro += __shfl_xor_sync(0xffffffffu, fro, 1);
  fro += __shfl_xor_sync(0xffffffffu, fro, 2);
  const T eps = teps<T>();
  const T tol2 = T(64) * eps * eps * fro;
  int done = -1;
  for (int sweep = 0; sweep <= max_sweeps; ++sweep) {
    T off = T(0);
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (c != l) off += abs2(Ar[c]);
    off += __shfl_xor_sync(0xffffffffu, off, 1);
    off += __shfl_xor_sync(0xffffffffu, off, 2);
    if (done < 0 && (off <= tol2 || fro == T(0))) done = sweep;
    if (__all_sync(0xffffffffu, done >= 0) || sweep == max_sweeps) break;
    const bool frozen = done >= 0;
    int rot = quad_round<1>(Ar, Vr, l, base, frozen);
    rot |= quad_round<2>(Ar, Vr, l, base, frozen);
    rot |= quad_round<3>(Ar, Vr, l, base, frozen);
    rot |= __shfl_xor_sync(0xffffffffu, rot, 1);
    rot |= __shfl_xor_sync(0xffffffffu, rot, 2);
    if (done < 0 && !rot) done = sweep + 1;
  }
  return done;
}

// Ascending order (stable) of the group's diagonal: lam[c] = A[c][c], ord[c] = the
// index of the c-th smallest.
template <typename T>
__device__ __forceinline__ void quad_order(const cx<T> (&Ar)[4], int l, int base, T (&lam)[4],
                                           int (&ord)[4]) {
  const T own = sel4(Ar, l).re;
#pragma unroll
  for (int c = 0; c < 4; ++c) lam[c] = __shfl_sync(0xffffffffu, own, base + c);
#pragma unroll
  for (int x = 0; x < 4; ++x) {
    int rk = 0;
#pragma unroll
    for (int y = 0; y < 4; ++y) rk += (lam[y] < lam[x]) || (lam[y] == lam[x] && y < x);
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (rk == c) ord[c] = x;
  }
}

__host__ __device__ inline TabShape tab_shape_split(int M) {
  int B = 1;
  while (B * B < M) ++B;
  return {B, (M + B - 1) / B};
}

__device__ inline void fill_tab_df(cdf* lo, cdf* hi, int M, TabShape t) {
  for (int m = threadIdx.x; m < t.B + t.H; m += blockDim.x) {
    const long long e = m < t.B ? m : (long long)(m - t.B) * t.B;
    double sn, cs;
    sincospi(2.0 * double(e) / double(M), &sn, &cs);
    *(m < t.B ? lo + m : hi + (m - t.B)) = cdf_from(z64(cs, sn));
  }
}

__device__ __forceinline__ cdf tab_at_df(const cdf* lo, const cdf* hi, TabShape t, int m) {
  return hi[m / t.B] * lo[m % t.B];
}

// acc += a b + c d with b and d exact in float (df_mac2 without the terms in their low parts).
__device__ __forceinline__ void df_mac2(df& acc, df a, float b, df c, float d) {
  const float p = a.hi * b, q = c.hi * d;
  const float e = fmaf(a.lo, b, fmaf(a.hi, b, -p)), f = fmaf(c.lo, d, fmaf(c.hi, d, -q));
  const df s = df_two_sum(p, q), t = df_two_sum(acc.hi, s.hi);
  acc = df_two_sum(t.hi, (s.lo + t.lo) + ((e + f) + acc.lo));
}

__device__ __forceinline__ df group_sum_df(df v) {
  v = df_sum(v, shfl_xor_df(v, 1));
  return df_sum(v, shfl_xor_df(v, 2));
}

__device__ __forceinline__ c32 group_sum_c32(c32 v) {
  v.re += __shfl_xor_sync(0xffffffffu, v.re, 1);
  v.im += __shfl_xor_sync(0xffffffffu, v.im, 1);
  v.re += __shfl_xor_sync(0xffffffffu, v.re, 2);
  v.im += __shfl_xor_sync(0xffffffffu, v.im, 2);
  return v;
}

// The refinement below is written with rolled loops and register selects rather
// than unrolled code: it runs once per k-point on few warps per SM, where a long
// straight-line body stalls on instruction fetch.

// (H x)[l] for an FP32 vector x held one entry per lane (x[q] in lane q).
__device__ __forceinline__ cdf quad_matvec(const cdf (&Hr)[4], c32 x, int base) {
  cdf acc = cdf_zero();
#pragma unroll 1
  for (int q = 0; q < 4; ++q) {
    const cdf h = sel4(Hr, q);
    const c32 v = shfl_z(x, base + q);
    df_mac2(acc.re, h.re, v.re, h.im, -v.im);
    df_mac2(acc.im, h.re, v.im, h.im, v.re);
  }
  return acc;
}

// An FP32 pair x0, x1 of the group with h_c = H x_c: the Ritz matrix g = x^dag h and the
// deviation e = x^dag x - I (~1e-7, kept in FP32; with kDev) from double-float sums.
struct QuadPair {
  df g00, g11, gre, gim;
  float e00, e11;
  c32 e01;
};
template <bool kDev>
__device__ __forceinline__ QuadPair quad_pair(c32 x0, c32 x1, cdf h0, cdf h1) {
  QuadPair r;
  r.e00 = r.e11 = 0.f;
  r.e01 = c32(0.f, 0.f);
#pragma unroll 1
  for (int t = 0; t < 3; ++t) {  // (0, 0), (0, 1), (1, 1)
    const c32 a = t == 2 ? x1 : x0, b = t == 0 ? x0 : x1;
    const cdf h = t == 0 ? h0 : h1;
    df gr(0.f), gi(0.f), er(0.f), ei(0.f);
    df_mac2(gr, h.re, a.re, h.im, a.im);
    gr = group_sum_df(gr);
    if (t == 1) {
      df_mac2(gi, h.im, a.re, h.re, -a.im);
      r.gre = gr;
      r.gim = group_sum_df(gi);
    }
    if (t == 0) r.g00 = gr;
    if (t == 2) r.g11 = gr;
    if constexpr (kDev) {
      df_mac2(er, df(b.re), a.re, df(b.im), a.im);
      er = group_sum_df(er);
      if (t == 1) {
        df_mac2(ei, df(b.im), a.re, df(b.re), -a.im);
        r.e01 = c32(er.hi, group_sum_df(ei).hi);
      }
      const float d = (er.hi - 1.f) + er.lo;
      if (t == 0) r.e00 = d;
      if (t == 2) r.e11 = d;
    }
  }
  return r;
}

// e - 3/4 e^2 of a Hermitian 2 x 2 deviation: (I + e)^{-1/2} = I - (e - 3/4 e^2) / 2 to second
// order (e^2 ~ 1e-13 would stay as the error otherwise).
__device__ __forceinline__ void dev_second_order(float& e00, float& e11, c32& e01) {
  const float q = abs2(e01), t = 1.f - 0.75f * (e00 + e11);
  e00 -= 0.75f * fmaf(e00, e00, q);
  e11 -= 0.75f * fmaf(e11, e11, q);
  e01 = t * e01;
}

// Eigenvalues lo <= hi of the pair's 2 x 2 Ritz matrix in the orthonormalised basis, to second
// order in the deviation: (I + e)^{-1/2} g (I + e)^{-1/2} + s = g - (e' g + g e') / 2 + e g e / 4 + s
// with e' = e - 3/4 e^2, s a small Hermitian correction (the small terms in FP32; the FP32 rotations
// leave e up to ~5e-6, so that e g e / 4 is worth 1e-11);
// (a + d) / 2 -+ sqrt(((a - d) / 2)^2 + |b|^2) in double-float.
__device__ __forceinline__ void quad_pair_edges(QuadPair r, float s00, float s11, c32 s01, df& lo, df& hi) {
  const c32 g(r.gre.hi, r.gim.hi);
  {
    const c32 m00 = r.g00.hi * c32(r.e00, 0.f) + g * conj(r.e01), m01 = r.g00.hi * r.e01 + r.e11 * g;
    const c32 m10 = r.e00 * conj(g) + r.g11.hi * conj(r.e01), m11 = conj(g) * r.e01 + r.g11.hi * c32(r.e11, 0.f);
    s00 += 0.25f * (r.e00 * m00.re + (r.e01 * m10).re);
    s11 += 0.25f * ((conj(r.e01) * m01).re + r.e11 * m11.re);
    s01 = s01 + 0.25f * (r.e00 * m01 + r.e01 * m11);
  }
  dev_second_order(r.e00, r.e11, r.e01);
  const float a = r.g00.hi, d = r.g11.hi, m = 0.5f * (a + d), x = g.re * r.e01.re + g.im * r.e01.im;
  const df aa = df_sum(r.g00, df(s00 - r.e00 * a - x)), dd = df_sum(r.g11, df(s11 - r.e11 * d - x));
  const float eh = 0.5f * (r.e00 + r.e11);
  const df bre = df_sum(r.gre, df(s01.re - eh * g.re - m * r.e01.re)), bim = df_sum(r.gim, df(s01.im - eh * g.im - m * r.e01.im));
  const df mean = 0.5f * df_sum(aa, dd), half = 0.5f * df_sum(aa, -dd);
  const df q = df_sqrt(df_fma(half, half, df_fma(bre, bre, bim * bim)));
  lo = df_sum(mean, -q);
  hi = df_sum(mean, q);
}

// Occupied pair of a four-band H(k) given as double-float rows (lane l holds row
// l): FP32 Jacobi on the float part of H, made exactly Hermitian; one Newton
// correction of the two lowest FP32 vectors q_c in the FP32 eigenbasis with the
// residual R = H q_c - q_c rho_c in double-float (q_c += z_a C_ac, C_ac = z_a^dag R_c /
// (rho_c - lam_a) over the unoccupied z_a); one second-order Lowdin step; the gap from
// double-float Ritz values of the FP32 pairs with the second-order shifts
// -+ C^dag (lam_a - rho_c) C (accurate whatever the splitting inside each pair).  Four
// matrix-vector products in all: the refined pair needs none of its own.  Every lane of the
// warp must call it (warp shuffles).  Returns the Jacobi
// sweeps used (-1: no convergence); Q0, Q1 are row l of the occupied vectors.
__device__ __forceinline__ int quad_df_occupied(const cdf (&Hr)[4], int l, int base, int max_sweeps,
                                                cdf& Q0, cdf& Q1, double& gap) {
  c32 Ar[4], Vr[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) Ar[c] = c32(Hr[c].re.hi, c == l ? 0.f : Hr[c].im.hi);
#pragma unroll
  for (int cc = 0; cc < 4; ++cc) {
    const c32 v(Hr[cc].re.hi, Hr[cc].im.hi);  // own row, column cc
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const c32 t = shfl_z(v, base + c);     // A[c][cc] from lane c
      if (cc == l && c < l) Ar[c] = conj(t);
    }
  }
  const int sweeps = quad_jacobi(Ar, Vr, l, base, max_sweeps);
  float lam[4];
  int ord[4];
  quad_order(Ar, l, base, lam, ord);
  const c32 q0 = sel4(Vr, ord[0]), q1 = sel4(Vr, ord[1]), z0 = sel4(Vr, ord[2]), z1 = sel4(Vr, ord[3]);
  const float lz0 = sel4(lam, ord[2]), lz1 = sel4(lam, ord[3]);
  cdf h[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) h[t] = cdf_zero();
#pragma unroll 1
  for (int t = 0; t < 4; ++t) {
    const cdf v = quad_matvec(Hr, t == 0 ? q0 : (t == 1 ? q1 : (t == 2 ? z0 : z1)), base);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (u == t) h[u] = v;
  }
  QuadPair oc = quad_pair<false>(q0, q1, h[0], h[1]);
  const QuadPair un = quad_pair<true>(z0, z1, h[2], h[3]);
  // residuals and coefficients C[a][c]
  auto resid = [](cdf hv, c32 q, df rho) {
    return c32(df_sum(hv.re, -(q.re * rho)).hi, df_sum(hv.im, -(q.im * rho)).hi);
  };
  const c32 r0 = resid(h[0], q0, oc.g00), r1 = resid(h[1], q1, oc.g11);
  auto coef = [](c32 z, c32 r, float den) {
    const c32 d = group_sum_c32(conj(z) * r);
    return den != 0.f ? (1.f / den) * d : c32(0.f, 0.f);
  };
  const float d00 = oc.g00.hi - lz0, d01 = oc.g11.hi - lz0, d10 = oc.g00.hi - lz1, d11 = oc.g11.hi - lz1;
  const c32 c00 = coef(z0, r0, d00), c01 = coef(z0, r1, d01), c10 = coef(z1, r0, d10), c11 = coef(z1, r1, d11);
  const c32 u0 = z0 * c00 + z1 * c10, u1 = z0 * c01 + z1 * c11;
  // z_a^dag q_c: the pairs are orthogonal to FP32 only, which counts at second order
  const c32 o00 = group_sum_c32(conj(z0) * q0), o01 = group_sum_c32(conj(z0) * q1);
  const c32 o10 = group_sum_c32(conj(z1) * q0), o11 = group_sum_c32(conj(z1) * q1);
  Q0 = cdf(df_two_sum(q0.re, u0.re), df_two_sum(q0.im, u0.im));
  Q1 = cdf(df_two_sum(q1.re, u1.re), df_two_sum(q1.im, u1.im));
  // Lowdin step: the deviation E of the corrected pair in double-float
  {
    float e00 = 0.f, e11 = 0.f;
    c32 e01(0.f, 0.f);
#pragma unroll 1
    for (int t = 0; t < 3; ++t) {  // (0, 0), (0, 1), (1, 1)
      const cdf xa = t == 2 ? Q1 : Q0, xb = t == 0 ? Q0 : Q1;
      cdf g = cdf_zero();
      cfma_conj(g, xa, xb);
      const df gre = group_sum_df(g.re);
      const float d = (gre.hi - 1.f) + gre.lo;
      if (t == 0) e00 = d;
      if (t == 1) e01 = c32(gre.hi, group_sum_df(g.im).hi);
      if (t == 2) e11 = d;
    }
    // the FP32 pair's own deviation, for its Ritz matrix: E - C^dag C - o^dag C - C^dag o
    oc.e00 = e00 - (conj(c00 + 2.f * o00) * c00).re - (conj(c10 + 2.f * o10) * c10).re;
    oc.e11 = e11 - (conj(c01 + 2.f * o01) * c01).re - (conj(c11 + 2.f * o11) * c11).re;
    oc.e01 = e01 - conj(c00 + o00) * c01 - conj(c10 + o10) * c11 - conj(c00) * o01 - conj(c10) * o11;
    dev_second_order(e00, e11, e01);
    const c32 x0(Q0.re.hi, Q0.im.hi), x1(Q1.re.hi, Q1.im.hi);
    const c32 f0 = e00 * x0 + x1 * conj(e01), f1 = x0 * e01 + e11 * x1;
    Q0 = cdf(df_sum(Q0.re, df(-0.5f * f0.re)), df_sum(Q0.im, df(-0.5f * f0.im)));
    Q1 = cdf(df_sum(Q1.re, df(-0.5f * f1.re)), df_sum(Q1.im, df(-0.5f * f1.im)));
  }
  // second-order shifts of the Ritz matrices (level repulsion between the pairs)
  df occ_lo, occ_hi, un_lo, un_hi;
  const float m0 = 0.5f * (d00 + d01), m1 = 0.5f * (d10 + d11);
  quad_pair_edges(oc, d00 * abs2(c00) + d10 * abs2(c10), d01 * abs2(c01) + d11 * abs2(c11),
                  m0 * (conj(c00) * c01) + m1 * (conj(c10) * c11), occ_lo, occ_hi);
  // (the unoccupied vectors' coefficients on the occupied ones are -conj(C + o))
  const c32 b00 = c00 + o00, b01 = c01 + o01, b10 = c10 + o10, b11 = c11 + o11;
  const float n0 = 0.5f * (d00 + d10), n1 = 0.5f * (d01 + d11);
  quad_pair_edges(un, -(d00 * abs2(b00) + d01 * abs2(b01)), -(d10 * abs2(b10) + d11 * abs2(b11)),
                  -(n0 * (b00 * conj(b10)) + n1 * (b01 * conj(b11))), un_lo, un_hi);
  gap = df_to_double(un_lo - occ_hi);
  return sweeps;
}

}  // namespace bw
