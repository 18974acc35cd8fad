// Few-band models (n = 2 or 4): Bloch Hamiltonian, occupied states and projected-spin
// sector in registers (Sec. I "exact diagonalization", Eq. 1, Sec. IV); one thread per
// k-point at n = 2, four lanes per k-point at n = 4.
//
// The matrix sizes are compile-time constants, loops unroll, and the arrays stay in
// registers.  The Bloch phases come from per-CTA
// tables: with an integer loop direction and an integer transverse direction,
// f(j, i).R = origin.R + j (loop.R) / N + i (trans.R) / N_t, so
// exp(i 2pi f.R) = exp(i 2pi origin.R) w_N^{(j loop.R) mod N} w_Nt^{(i trans.R) mod N_t}
// with w_M = exp(i 2pi / M) tabulated once per CTA (in two levels for long grids).
#include <float.h>

#include <cstring>
#include <type_traits>

#include "launch.h"
#include "quad.cuh"

namespace bw {
namespace {

// Serial cyclic Jacobi on a Hermitian NN x NN matrix held in registers; V collects
// the rotations (same rotation formula and skip test as the block solver).  Returns the sweeps
// used or -1 without convergence.
template <int NN, typename T>
__device__ __forceinline__ int jac_serial(cx<T> (&A)[NN][NN], cx<T> (&V)[NN][NN], int max_sweeps) {
#pragma unroll
  for (int r = 0; r < NN; ++r)
#pragma unroll
    for (int c = 0; c < NN; ++c) V[r][c] = cx<T>(T(r == c), T(0));
  T fro = T(0);
#pragma unroll
  for (int r = 0; r < NN; ++r)
#pragma unroll
    for (int c = 0; c < NN; ++c) fro += abs2(A[r][c]);
  const T tol2 = T(64) * teps<T>() * teps<T>() * fro;
  for (int sweep = 0; sweep <= max_sweeps; ++sweep) {
    T off = T(0);
#pragma unroll
    for (int p = 0; p < NN; ++p)
#pragma unroll
      for (int q = p + 1; q < NN; ++q) off += T(2) * abs2(A[p][q]);
    if (off <= tol2 || fro == T(0)) return sweep;
    if (sweep == max_sweeps) break;
    bool rotated = false;
#pragma unroll
    for (int p = 0; p < NN; ++p)
#pragma unroll
      for (int q = p + 1; q < NN; ++q) {
        const cx<T> b = A[p][q];
        const T a = A[p][p].re, d = A[q][q].re;
        T c, t, ab;
        cx<T> sc;
        if (!quad_angle(a, d, b, c, sc, t, ab)) continue;
        rotated = true;
#pragma unroll
        for (int k = 0; k < NN; ++k) {
          const cx<T> ap = A[p][k], aq = A[q][k];
          A[p][k] = c * ap - sc * aq;
          A[q][k] = conj(sc) * ap + c * aq;
        }
#pragma unroll
        for (int k = 0; k < NN; ++k) {
          const cx<T> ap = A[k][p], aq = A[k][q];
          A[k][p] = c * ap - aq * conj(sc);
          A[k][q] = ap * sc + c * aq;
          const cx<T> vp = V[k][p], vq = V[k][q];
          V[k][p] = c * vp - vq * conj(sc);
          V[k][q] = vp * sc + c * vq;
        }
        A[p][q] = cx<T>(T(0), T(0));
        A[q][p] = cx<T>(T(0), T(0));
        A[p][p] = cx<T>(a - t * ab, T(0));
        A[q][q] = cx<T>(d + t * ab, T(0));
      }
    if (!rotated) return sweep + 1;
  }
  return -1;
}

// Columns of V sorted by ascending diagonal of A (stable): Vs[:, c], lam[c].
template <int NN, typename T>
__device__ __forceinline__ void sort_eig(const cx<T> (&A)[NN][NN], const cx<T> (&V)[NN][NN],
                                         cx<T> (&Vs)[NN][NN], T (&lam)[NN]) {
  int rank[NN];
#pragma unroll
  for (int a = 0; a < NN; ++a) {
    int r = 0;
#pragma unroll
    for (int b = 0; b < NN; ++b)
      r += (A[b][b].re < A[a][a].re) || (A[b][b].re == A[a][a].re && b < a);
    rank[a] = r;
  }
#pragma unroll
  for (int c = 0; c < NN; ++c) {
#pragma unroll
    for (int a = 0; a < NN; ++a)
      if (rank[a] == c) {
        lam[c] = A[a][a].re;
#pragma unroll
        for (int r = 0; r < NN; ++r) Vs[r][c] = V[r][a];
      }
  }
}

constexpr int TINY_THREADS = 128;
// Above this many points a direction's phase table is split in two levels
// (w^m = w^{B (m / B)} w^{m mod B}, B ~ sqrt(M)): each CTA fills its own tables, and past
// about a hundred entries their sines and cosines (~45 FP64 instructions each) would cost
// more than the extra product per translation (N_t = 512: a quarter of the kernel).
constexpr int TAB_SPLIT = 64;

__host__ __device__ inline TabShape tab_shape(int M) {
  if (M <= TAB_SPLIT) return {M, 0};
  int B = 1;
  while (B * B < M) ++B;
  return {B, (M + B - 1) / B};
}

__device__ __forceinline__ z64 tab_at(const z64* lo, const z64* hi, TabShape t, int m) {
  if (t.H == 0) return lo[m];
  return hi[m / t.B] * lo[m % t.B];
}

// Eigenvalues lo <= hi of the Hermitian 2 x 2 matrix [[a, b], [conj b, d]] and the unit
// eigenvector (v0, v1) of lo; that of hi is (-conj v1, conj v0).  With half = (a - d) / 2
// and r = sqrt(half^2 + |b|^2) the vector is (-b, half + r) or (r - half, -conj b),
// whichever has the sum of two positive terms in it.
__device__ __forceinline__ void eig2_herm(double a, double d, z64 b, double& lo, double& hi, z64& v0, z64& v1) {
  const double mid = 0.5 * (a + d), half = 0.5 * (a - d);
  const double r = sqrt(fma(half, half, abs2(b)));
  lo = mid - r;
  hi = mid + r;
  const double g = fabs(half) + r, nn = fma(g, g, abs2(b));
  if (!(nn > 0.0)) {
    v0 = z64(1.0, 0.0);
    v1 = z64(0.0, 0.0);
    return;
  }
  const double inv = rsqrt(nn);
  const z64 bs(inv * b.re, inv * b.im);
  v0 = half >= 0.0 ? z64(-bs.re, -bs.im) : z64(inv * g, 0.0);
  v1 = half >= 0.0 ? z64(inv * g, 0.0) : z64(-bs.re, bs.im);
}

// j q mod M for 0 <= j, q < M: 32-bit arithmetic while the product fits.
__device__ __forceinline__ unsigned mulmod(unsigned j, unsigned q, unsigned M) {
  return M <= 65536u ? j * q % M : unsigned((unsigned long long)j * q % M);
}

// Shared-memory tables of a few-band CTA with `slots` k-points: Bloch phases of the
// translations per k-point, the phase tables of an integer plane, and the hopping list
// when it is short (an L2 round trip per hopping otherwise).
struct TinySmem {
  z64 *cache, *tabN, *tabNt, *oph, *ht;
  int *lR, *tR, *sR, *hr;
};

constexpr int TINY_PLAN_MAX = 1024;  // hoppings staged in shared memory

__host__ __device__ inline size_t tiny_smem_bytes(int nR, int n_hop, int slots, bool use_tab, TabShape tN,
                                                  TabShape tT) {
  size_t b = size_t(nR) * slots * sizeof(z64);
  if (use_tab) b += (size_t(tN.B) + tN.H + tT.B + tT.H + nR) * sizeof(z64) + 3 * size_t(nR) * sizeof(int);
  if (n_hop <= TINY_PLAN_MAX) b += size_t(n_hop) * (sizeof(z64) + sizeof(int));
  return b;
}

// Carves the tables out of `smem` and fills everything but the per-k-point phases; eb / ee:
// the hopping range of entry (r, c) of the NN x NN matrix (empty where the list has none).
template <int NN>
__device__ __forceinline__ TinySmem tiny_tables(const StatesArgs& a, unsigned char* smem, int slots, bool use_tab,
                                                int* eb, int* ee) {
  const DevModel& md = a.model;
  const int tid = threadIdx.x, bd = blockDim.x, nR = md.n_R, N = a.plane.N, Nt = a.plane.N_t;
  const bool plan = md.n_hop <= TINY_PLAN_MAX;
  const TabShape tN = tab_shape(N), tT = tab_shape(Nt);
  TinySmem S;
  S.cache = reinterpret_cast<z64*>(smem);
  S.tabN = S.cache + nR * slots;
  S.tabNt = S.tabN + (use_tab ? tN.B + tN.H : 0);
  S.oph = S.tabNt + (use_tab ? tT.B + tT.H : 0);
  S.ht = S.oph + (use_tab ? nR : 0);
  S.lR = reinterpret_cast<int*>(S.ht + (plan ? md.n_hop : 0));
  S.tR = S.lR + (use_tab ? nR : 0);
  S.sR = S.tR + (use_tab ? nR : 0);
  S.hr = S.sR + (use_tab ? nR : 0);
  for (int e = tid; e < NN * NN; e += bd) eb[e] = ee[e] = 0;
  if (plan)
    for (int h = tid; h < md.n_hop; h += bd) {
      S.ht[h] = md.hop_t[h];
      S.hr[h] = md.hop_r[h];
    }
  if (use_tab) {
    // w_N^m, w_Nt^m (both levels) and the translations' factors at the origin: one loop, so
    // that a CTA with a thread per entry evaluates sine and cosine (~40 dependent FP64
    // operations) once
    const int cN = tN.B + tN.H, cT = tT.B + tT.H;
    for (int m = tid; m < cN + cT + nR; m += bd) {
      double x = 0.0;
      if (m < cN + cT) {
        const int q = m < cN ? m : m - cN, M = m < cN ? N : Nt;
        const TabShape t = m < cN ? tN : tT;
        x = 2.0 * double(q < t.B ? (long long)q : (long long)(q - t.B) * t.B) / double(M);
      } else {
        const int r = m - cN - cT;
        const int* R = md.Rv + 3 * r;
        long long l = 0, t = 0, sw = 0;
        for (int d = 0; d < 3; ++d) {
          x += a.plane.origin[d] * double(R[d]);
          l += (long long)(a.plane.loop_dir[d]) * R[d];
          t += (long long)(a.plane.trans_dir[d]) * R[d];
          sw += (long long)a.plane.sweep[d] * R[d];
        }
        x *= 2.0;
        // exponents of w_N per loop step, and of w_Nt per transverse and per sweep step
        S.lR[r] = pmod(l, N);
        S.tR[r] = pmod(a.plane.N_s > 1 ? t * a.plane.N_s : t, Nt);
        S.sR[r] = pmod(a.plane.N_s > 1 ? sw * a.plane.N_tp : 0, Nt);
      }
      double sn, cs;
      sincospi(x, &sn, &cs);
      S.tabN[m] = z64(cs, sn);  // tabN, tabNt and oph follow each other
    }
  }
  if (!plan) {
    S.ht = const_cast<z64*>(md.hop_t);
    S.hr = const_cast<int*>(md.hop_r);
  }
  __syncthreads();
  for (int e = tid; e < md.n_ent; e += bd) {
    const int at = md.ent_row[e] * NN + md.ent_col[e];
    eb[at] = md.ent_start[e];
    ee[at] = md.ent_start[e + 1];
  }
  __syncthreads();
  return S;
}

// Bloch phases at k-point k into slot `slot` of S.cache: translations first, first + step, ...
__device__ __forceinline__ void tiny_phases(const StatesArgs& a, const TinySmem& S, long long k, int slot, int slots,
                                            bool use_tab, int first, int step) {
  const int nR = a.model.n_R, N = a.plane.N, Nt = a.plane.N_t;
  if (use_tab || !a.f) {
    const int i = int(k / N), j = int(k - (long long)i * N);
    if (use_tab) {
      const TabShape tN = tab_shape(N), tT = tab_shape(Nt);
      const int s = a.plane.N_s > 1 ? i / a.plane.N_tp : 0, it = a.plane.N_s > 1 ? i - s * a.plane.N_tp : i;
      for (int r = first; r < nR; r += step) {
        const int mN = int(mulmod(j, S.lR[r], N));
        int mT = int(mulmod(it, S.tR[r], Nt));
        if (a.plane.N_s > 1) {
          mT += int(mulmod(s, S.sR[r], Nt));
          if (mT >= Nt) mT -= Nt;
        }
        S.cache[r * slots + slot] =
            S.oph[r] * tab_at(S.tabN, S.tabN + tN.B, tN, mN) * tab_at(S.tabNt, S.tabNt + tT.B, tT, mT);
      }
    } else {
      double f[3];
      plane_f(a.plane, i, j, f);
      for (int r = first; r < nR; r += step) S.cache[r * slots + slot] = bloch_phase(f, a.model.Rv + 3 * r);
    }
  } else {
    const double f[3] = {a.f[3 * k], a.f[3 * k + 1], a.f[3 * k + 2]};
    for (int r = first; r < nR; r += step) S.cache[r * slots + slot] = bloch_phase(f, a.model.Rv + 3 * r);
  }
}

// Entry of H(k) from its hopping range.
__device__ __forceinline__ z64 tiny_entry(const TinySmem& S, int h0, int h1, int slot, int slots) {
  z64 acc(0.0, 0.0);
  for (int h = h0; h < h1; ++h) cfma(acc, S.ht[h], S.cache[S.hr[h] * slots + slot]);
  return acc;
}

// Sector columns of the projected spin operator from its eigenvalues mu (ascending): the
// checks, the outputs and the first column c0 of the sector.
template <int PP>
__device__ __forceinline__ int tiny_sector(const StatesArgs& a, long long k, const double (&mu)[PP], bool ok,
                                           bool write) {
  int neg = 0;
  double g = INFINITY;
#pragma unroll
  for (int c = 0; c < PP; ++c) {
    neg += mu[c] < 0.0;
    g = fmin(g, fabs(mu[c]));
    if (a.pso_evals && write) a.pso_evals[k * PP + c] = mu[c];
  }
  if (a.pso_median) {
    neg = PP / 2;
    g = mu[PP / 2] - mu[PP / 2 - 1];
  }
  if (write) {
    if (a.pso_gap) a.pso_gap[k] = g;
    if (!ok) report(a.status, ST_ENOCONV, k, 0.0);
    if (neg != PP / 2 || !(g > a.pso_gap_tol)) report(a.status, ST_EPSOGAP, k, g);
  }
  return a.sign < 0 ? 0 : PP / 2;
}

// Columns v of the sector in the occupied basis from the projected spin operator S (Hermitian,
// overwritten), with the checks and outputs of tiny_sector.
template <int PP>
__device__ __forceinline__ void tiny_sector_columns(const StatesArgs& a, long long k, z64 (&S)[PP][PP], bool write,
                                                    z64 (&v)[PP][PP / 2]) {
  double mu[PP];
  if constexpr (PP == 2) {
    z64 v0, v1;
    eig2_herm(S[0][0].re, S[1][1].re, S[0][1], mu[0], mu[1], v0, v1);
    const bool up = tiny_sector<2>(a, k, mu, true, write) != 0;
    v[0][0] = up ? -conj(v1) : v0;
    v[1][0] = up ? conj(v0) : v1;
  } else {
    z64 SV[PP][PP], SVs[PP][PP];
    const bool okp = jac_serial<PP, double>(S, SV, a.max_sweeps) >= 0;
    sort_eig<PP, double>(S, SV, SVs, mu);
    const bool up = tiny_sector<PP>(a, k, mu, okp, write) != 0;
#pragma unroll
    for (int q = 0; q < PP; ++q)
#pragma unroll
      for (int c = 0; c < PP / 2; ++c) v[q][c] = up ? SVs[q][c + PP / 2] : SVs[q][c];
  }
}

// The plan arrays in the kernel's parameter copy of the plan instead of at dbase.
__device__ __forceinline__ void tiny_relocate(StatesArgs& a, const unsigned char* inl, const char* dbase) {
  auto at = [&](auto*& p) {
    if (p) p = reinterpret_cast<std::remove_reference_t<decltype(p)>>(inl + (reinterpret_cast<const char*>(p) - dbase));
  };
  at(a.model.Rv);
  at(a.model.ent_row);
  at(a.model.ent_col);
  at(a.model.ent_start);
  at(a.model.hop_r);
  at(a.model.hop_t);
  if (a.op.nnz > 0) {
    at(a.op.row);
    at(a.op.col);
    at(a.op.val);
  }
}

// n = 2: one thread per k-point, eigenvalues and states in closed form.
template <int PP>
__device__ __forceinline__ void states_two(const StatesArgs& a, int use_tab) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int eb[4], ee[4];
  const int tid = threadIdx.x, bd = blockDim.x;
  const TinySmem T = tiny_tables<2>(a, smem, bd, use_tab != 0, eb, ee);
  const long long k = (long long)blockIdx.x * bd + tid;
  if (k >= a.K) return;
  tiny_phases(a, T, k, tid, bd, use_tab != 0, 0, 1);
  const double h00 = tiny_entry(T, eb[0], ee[0], tid, bd).re, h11 = tiny_entry(T, eb[3], ee[3], tid, bd).re;
  const z64 h01 = tiny_entry(T, eb[1], ee[1], tid, bd);
  double lo, hi;
  z64 Q[2][2];
  eig2_herm(h00, h11, h01, lo, hi, Q[0][0], Q[1][0]);
  Q[0][1] = -conj(Q[1][0]);
  Q[1][1] = conj(Q[0][0]);
  const double gap = PP < 2 ? hi - lo : INFINITY;
  a.gap[k] = gap;
  if (!(gap > a.gap_tol)) report(a.status, ST_EGAP, k, gap);
  z64* out = a.U + k * 2LL * (a.op.nnz > 0 ? PP / 2 : PP);
  if (a.op.nnz > 0) {
    if constexpr (PP == 2) {
      // projected spin operator restricted to the occupied space (Sec. IV)
      z64 S[2][2] = {};
      for (int q = 0; q < a.op.nnz; ++q) {
        const bool r1 = a.op.row[q] != 0, c1 = a.op.col[q] != 0;
        const z64 v = a.op.val[q];
#pragma unroll
        for (int x = 0; x < 2; ++x)
#pragma unroll
          for (int y = 0; y < 2; ++y) cfma_conj(S[x][y], r1 ? Q[1][x] : Q[0][x], v * (c1 ? Q[1][y] : Q[0][y]));
      }
      double mu[2];
      z64 v0, v1;
      eig2_herm(S[0][0].re, S[1][1].re, 0.5 * (S[0][1] + conj(S[1][0])), mu[0], mu[1], v0, v1);
      if (tiny_sector<2>(a, k, mu, true, true)) {
        const z64 t = -conj(v1);
        v1 = conj(v0);
        v0 = t;
      }
#pragma unroll
      for (int r = 0; r < 2; ++r) out[r] = Q[r][0] * v0 + Q[r][1] * v1;
    }
  } else {
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int c = 0; c < PP; ++c) out[r * PP + c] = Q[r][c];
  }
}

// ---------------------------------------------------------------------------
// n = 4, four lanes per k-point, to FP64 accuracy: lane l of a group of four consecutive
// lanes holds row l of H(k) and entry l of every vector (quad.cuh).
// ---------------------------------------------------------------------------
constexpr int QUAD_THREADS = 128;  // 32 k-points per CTA

__device__ __forceinline__ z64 quad_sum(z64 v) {
  v.re += __shfl_xor_sync(0xffffffffu, v.re, 1);
  v.im += __shfl_xor_sync(0xffffffffu, v.im, 1);
  v.re += __shfl_xor_sync(0xffffffffu, v.re, 2);
  v.im += __shfl_xor_sync(0xffffffffu, v.im, 2);
  return v;
}
__device__ __forceinline__ double quad_sum(double v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v + __shfl_xor_sync(0xffffffffu, v, 2);
}

// Sums of four doubles over the group, in every lane: each lane adds up one of them (3 FP64
// additions per lane instead of 8) and the results are shuffled back.
__device__ __forceinline__ void quad_sum4(double& v0, double& v1, double& v2, double& v3, int l, int base) {
  const bool b1 = l & 2, b0 = l & 1;
  const double k0 = (b1 ? v2 : v0) + __shfl_xor_sync(0xffffffffu, b1 ? v0 : v2, 2);
  const double k1 = (b1 ? v3 : v1) + __shfl_xor_sync(0xffffffffu, b1 ? v1 : v3, 2);
  const double t = (b0 ? k1 : k0) + __shfl_xor_sync(0xffffffffu, b0 ? k0 : k1, 1);
  v0 = __shfl_sync(0xffffffffu, t, base);
  v1 = __shfl_sync(0xffffffffu, t, base + 1);
  v2 = __shfl_sync(0xffffffffu, t, base + 2);
  v3 = __shfl_sync(0xffffffffu, t, base + 3);
}

// X^dag Y of the group's vectors, every lane receiving the (Hermitian) result.
template <int KK>
__device__ __forceinline__ void quad_gram(const z64 (&X)[KK], const z64 (&Y)[KK], z64 (&G)[KK][KK], int l, int base) {
  if constexpr (KK == 2) {
    double d0 = fma(X[0].re, Y[0].re, X[0].im * Y[0].im), d1 = fma(X[1].re, Y[1].re, X[1].im * Y[1].im);
    z64 g(0.0, 0.0);
    cfma_conj(g, X[0], Y[1]);
    quad_sum4(d0, d1, g.re, g.im, l, base);
    G[0][0] = z64(d0, 0.0);
    G[1][1] = z64(d1, 0.0);
    G[0][1] = g;
    G[1][0] = conj(g);
  } else {
#pragma unroll
    for (int x = 0; x < KK; ++x)
#pragma unroll
      for (int y = x; y < KK; ++y) {
        if (x == y) {
          G[x][x] = z64(quad_sum(fma(X[x].re, Y[x].re, X[x].im * Y[x].im)), 0.0);
        } else {
          z64 g(0.0, 0.0);
          cfma_conj(g, X[x], Y[y]);
          G[x][y] = quad_sum(g);
          G[y][x] = conj(G[x][y]);
        }
      }
  }
}

template <int KK>
__device__ __forceinline__ void quad_apply(const z64 (&Hr)[4], const z64 (&X)[KK], z64 (&HX)[KK], int base) {
#pragma unroll
  for (int c = 0; c < KK; ++c) {
    HX[c] = z64(0.0, 0.0);
#pragma unroll
    for (int q = 0; q < 4; ++q) cfma(HX[c], Hr[q], shfl_z(X[c], base + q));
  }
}

// E = X^dag X - I, formed in FP64; the vectors are orthonormal to FP32 or better, so E
// itself is kept in FP32.
template <int KK>
__device__ __forceinline__ void quad_dev(const z64 (&X)[KK], c32 (&E)[KK][KK], int l, int base) {
  z64 G[KK][KK];
  quad_gram<KK>(X, X, G, l, base);
#pragma unroll
  for (int x = 0; x < KK; ++x)
#pragma unroll
    for (int y = x; y < KK; ++y) {
      E[x][y] = x == y ? c32(float(G[x][x].re - 1.0), 0.f) : ccast<float>(G[x][y]);
      if (x != y) E[y][x] = conj(E[x][y]);
    }
}

// First-order Lowdin step X <- X - X E / 2 (an error of 6e-8 E, which the next step or
// quad_dev_correct removes: E is ~1e-7 in the first step and ~1e-13 in the last).
template <int KK>
__device__ __forceinline__ void quad_lowdin(z64 (&X)[KK], const c32 (&E)[KK][KK]) {
  c32 x32[KK];
#pragma unroll
  for (int c = 0; c < KK; ++c) x32[c] = ccast<float>(X[c]);
#pragma unroll
  for (int c = 0; c < KK; ++c) {
    c32 d(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < KK; ++q) cfma(d, x32[q], E[q][c]);
    X[c] = z64(X[c].re - 0.5 * double(d.re), X[c].im - 0.5 * double(d.im));
  }
}

// Ritz matrix of the orthonormalised vectors from that of vectors with a deviation
// E <~ 1e-12: G - (E G + G E) / 2, the small terms in FP32.
template <int KK>
__device__ __forceinline__ void quad_dev_correct(z64 (&G)[KK][KK], const c32 (&E)[KK][KK]) {
  c32 g[KK][KK];
#pragma unroll
  for (int x = 0; x < KK; ++x)
#pragma unroll
    for (int y = 0; y < KK; ++y) g[x][y] = ccast<float>(G[x][y]);
#pragma unroll
  for (int x = 0; x < KK; ++x)
#pragma unroll
    for (int y = x; y < KK; ++y) {
      c32 d(0.f, 0.f);
#pragma unroll
      for (int q = 0; q < KK; ++q) {
        cfma(d, E[x][q], g[q][y]);
        cfma(d, g[x][q], E[q][y]);
      }
      G[x][y] = z64(G[x][y].re - 0.5 * double(d.re), x == y ? 0.0 : G[x][y].im - 0.5 * double(d.im));
      if (x != y) G[y][x] = conj(G[x][y]);
    }
}

// Largest (want_max) or smallest eigenvalue of a small Hermitian matrix.
template <int KK>
__device__ __forceinline__ double herm_edge(z64 (&G)[KK][KK], bool want_max) {
  if constexpr (KK == 1) {
    return G[0][0].re;
  } else {
    z64 V[KK][KK];
    jac_serial<KK, double>(G, V, 60);
    double e = G[0][0].re;
#pragma unroll
    for (int c = 1; c < KK; ++c) e = want_max ? fmax(e, G[c][c].re) : fmin(e, G[c][c].re);
    return e;
  }
}

// Occupied block (the lowest PP < 4 states; Q: row l) and direct gap of the group's H to FP64
// accuracy without an FP64 eigensolve: FP32 Jacobi gives a start with an error of
// e0 ~ 1e-7 ||H|| / gap; the first correction squares it, and each further one, in the same FP32
// vectors, multiplies it by about e0,
//   Q <- Q + Z C,  C[a][c] = z_a^dag (H Q - Q G)_c / (G_cc - lam_a),  G = Q^dag H Q,
// (z_a, lam_a the unoccupied FP32 pairs).  The products that decide the accuracy (H Q, G,
// the residual, the Gram matrices) are FP64; C and the correction, which only have to be
// right relative to their own small size, are FP32.  Two corrections are the rule: the loop ends
// when |C| <= 3e-9, which leaves |C| e0 <= 3e-16 ||H|| / gap, the forward error of an FP64
// eigensolver.
// The gap comes from the FP64 Ritz values of Q and of its orthogonal complement.
// Every lane of the warp must call it.  Returns false for a group where the method does not
// apply (the caller solves it in FP64): a gap below 1e-3 of the spectral radius, H outside
// the FP32 range, no convergence.
template <int PP>
__device__ __forceinline__ bool quad_refined(const z64 (&Hr)[4], int l, int base, int max_sweeps, z64 (&Q)[PP],
                                             double& gap) {
  constexpr int NU = 4 - PP;
  c32 Ar[4], Vr[4];
  float big = 0.f;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    Ar[c] = ccast<float>(Hr[c]);
    if (c == l) Ar[c].im = 0.f;
    big = fmaxf(big, fmaxf(fabsf(Ar[c].re), fabsf(Ar[c].im)));
  }
  big = fmaxf(big, __shfl_xor_sync(0xffffffffu, big, 1));
  big = fmaxf(big, __shfl_xor_sync(0xffffffffu, big, 2));
  bool ok = big > 1e-8f && big < 1e12f;
#pragma unroll
  for (int c = 0; c < 4; ++c)
    if (!ok) Ar[c] = c32(float(c), 0.f);  // keeps the group's sweeps finite
  ok = quad_jacobi(Ar, Vr, l, base, max_sweeps) >= 0 && ok;
  float lam[4];
  int ord[4];
  quad_order(Ar, l, base, lam, ord);
  c32 z[NU];
  float lu[NU];
#pragma unroll
  for (int c = 0; c < PP; ++c) Q[c] = ccast<double>(sel4(Vr, ord[c]));
#pragma unroll
  for (int c = 0; c < NU; ++c) {
    z[c] = sel4(Vr, ord[PP + c]);
    lu[c] = sel4(lam, ord[PP + c]);
  }
  const float lmin = sel4(lam, ord[0]), lmax = sel4(lam, ord[3]);
  ok = ok && lu[0] - sel4(lam, ord[PP - 1]) > 1e-3f * fmaxf(fabsf(lmin), fabsf(lmax));
  if (__all_sync(0xffffffffu, !ok)) return false;
  {
    c32 E[PP][PP];
    quad_dev<PP>(Q, E, l, base);
    quad_lowdin<PP>(Q, E);
  }
  z64 Go[PP][PP];
  bool done = false;
#pragma unroll 1
  for (int it = 0; it < 4; ++it) {
    if (__all_sync(0xffffffffu, done || !ok)) break;
    z64 HQ[PP], G[PP][PP];
    quad_apply<PP>(Hr, Q, HQ, base);
    quad_gram<PP>(Q, HQ, G, l, base);
    c32 R[PP], upd[PP];
#pragma unroll
    for (int c = 0; c < PP; ++c) {
      z64 acc = HQ[c];
#pragma unroll
      for (int q = 0; q < PP; ++q) cfms(acc, Q[q], G[q][c]);
      R[c] = ccast<float>(acc);
      upd[c] = c32(0.f, 0.f);
    }
    float c2 = 0.f;
#pragma unroll
    for (int a = 0; a < NU; ++a)
#pragma unroll
      for (int c = 0; c < PP; ++c) {
        c32 d = group_sum_c32(conj(z[a]) * R[c]);
        d = (1.f / (float(G[c][c].re) - lu[a])) * d;
        c2 += abs2(d);
        cfma(upd[c], z[a], d);
      }
    const bool step = !done;  // (a finished group only keeps the others of its warp company)
    if (step) {
      ok = ok && c2 < 1e-4f;
      done = c2 <= 1e-17f;
#pragma unroll
      for (int c = 0; c < PP; ++c) {
        Q[c] = z64(Q[c].re + double(upd[c].re), Q[c].im + double(upd[c].im));
#pragma unroll
        for (int q = 0; q < PP; ++q) Go[c][q] = G[c][q];
      }
    }
    // |C|^2 is what the correction takes from orthonormality; below 1e-12 the last
    // quad_lowdin and quad_dev_correct make up for it
    const bool ortho = step && c2 > 1e-12f;
    if (__any_sync(0xffffffffu, ortho)) {
      c32 E[PP][PP];
      z64 X[PP];
      quad_dev<PP>(Q, E, l, base);
#pragma unroll
      for (int c = 0; c < PP; ++c) X[c] = Q[c];
      quad_lowdin<PP>(X, E);
#pragma unroll
      for (int c = 0; c < PP; ++c)
        if (ortho) Q[c] = X[c];
    }
  }
  ok = ok && done;
  {
    c32 E[PP][PP];
    quad_dev<PP>(Q, E, l, base);
    quad_lowdin<PP>(Q, E);
    quad_dev_correct<PP>(Go, E);
  }
  // the unoccupied FP32 vectors, made orthogonal to Q and orthonormal in FP64
  z64 Z[NU], HZ[NU], Gu[NU][NU];
#pragma unroll
  for (int a = 0; a < NU; ++a) {
    const z64 za = ccast<double>(z[a]);
    Z[a] = za;
    z64 d[PP];
#pragma unroll
    for (int c = 0; c < PP; ++c) {
      d[c] = z64(0.0, 0.0);
      cfma_conj(d[c], Q[c], za);
    }
    if constexpr (PP == 2) {
      quad_sum4(d[0].re, d[0].im, d[1].re, d[1].im, l, base);
    } else {
#pragma unroll
      for (int c = 0; c < PP; ++c) d[c] = quad_sum(d[c]);
    }
#pragma unroll
    for (int c = 0; c < PP; ++c) cfms(Z[a], Q[c], d[c]);
  }
  {
    c32 E[NU][NU];
    quad_dev<NU>(Z, E, l, base);
    quad_lowdin<NU>(Z, E);
    quad_dev<NU>(Z, E, l, base);
    quad_apply<NU>(Hr, Z, HZ, base);
    quad_gram<NU>(Z, HZ, Gu, l, base);
    quad_dev_correct<NU>(Gu, E);
  }
  if constexpr (PP == 2) {  // one square root for both edges: even lanes the occupied one
    const bool un = l & 1;
    const double a0 = un ? Gu[0][0].re : Go[0][0].re, d0 = un ? Gu[1][1].re : Go[1][1].re;
    const double bre = un ? Gu[0][1].re : Go[0][1].re, bim = un ? Gu[0][1].im : Go[0][1].im;
    const double half = 0.5 * (a0 - d0), r = sqrt(fma(half, half, fma(bre, bre, bim * bim)));
    const double e = 0.5 * (a0 + d0) + (un ? -r : r), o = __shfl_xor_sync(0xffffffffu, e, 1);
    gap = un ? e - o : o - e;
  } else {
    gap = herm_edge<NU>(Gu, false) - herm_edge<PP>(Go, true);
  }
  return ok;
}

// FP64 instructions bound this kernel on large grids (a warp instruction occupies the pipe of
// an SM for ~19 clocks: ~450 per lane at p = 2) and instruction latency on small ones.
// Measured against FP64 Jacobi sweeps: Eq. 9 model, 32 x 32 x 16, 220 -> 93 us (one thread
// per k-point before); spin-Hall with the spin split, 51 x 51, 169 -> 47 us; the same refined
// solve with one thread per k-point 180 and 120 us (17 500 instructions in one warp per SM).
// The mixed-precision request takes it as well where the double-float kernel below does not
// apply.
template <int PP>
__device__ __forceinline__ void states_quad(const StatesArgs& a, int use_tab) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int eb[16], ee[16];
  constexpr int KPB = QUAD_THREADS / 4;
  const TinySmem T = tiny_tables<4>(a, smem, KPB, use_tab != 0, eb, ee);
  const int tid = threadIdx.x, l = tid & 3, kl = tid >> 2, base = (tid & 31) & ~3;
  const long long kraw = (long long)blockIdx.x * KPB + kl;
  const bool active = kraw < a.K;
  const long long k = active ? kraw : a.K - 1;  // idle groups recompute the last k-point
  tiny_phases(a, T, k, kl, KPB, use_tab != 0, l, 4);
  __syncwarp();
  // row l of H(k)
  // (each off-diagonal pair formed once: lane l makes (l, l + 1) and (l, l + 2) mod 4)
  z64 Hr[4];
  {
    const int c1 = (l + 1) & 3, c2 = (l + 2) & 3, c3 = (l + 3) & 3;
    double dg = 0.0;
    for (int h = eb[5 * l]; h < ee[5 * l]; ++h) {
      const z64 t = T.ht[h], w = T.cache[T.hr[h] * KPB + kl];
      dg = fma(t.re, w.re, fma(-t.im, w.im, dg));
    }
    const z64 s1 = tiny_entry(T, eb[4 * l + c1], ee[4 * l + c1], kl, KPB);
    const z64 s2 = tiny_entry(T, eb[4 * l + c2], ee[4 * l + c2], kl, KPB);
    const z64 s3 = conj(shfl_z(s1, base + c3)), t2 = shfl_z(s2, base + (l & 1));
#pragma unroll
    for (int c = 0; c < 4; ++c)
      Hr[c] = a.scale * (c == l ? z64(dg, 0.0) : (c == c1 ? s1 : (c == c3 ? s3 : (l < 2 ? t2 : conj(t2)))));
  }
  z64 Q[PP];
  double gap = INFINITY;
  bool ok = true, solved = false;
  if constexpr (PP < 4) solved = quad_refined<PP>(Hr, l, base, a.max_sweeps, Q, gap);
  if (!__all_sync(0xffffffffu, solved)) {  // FP64 Jacobi for the groups that need it
    z64 Ar[4], Vr[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) Ar[c] = solved ? z64(0.0, 0.0) : Hr[c];
    const int sweeps = quad_jacobi(Ar, Vr, l, base, a.max_sweeps);
    double lam[4];
    int ord[4];
    quad_order(Ar, l, base, lam, ord);
    if (!solved) {
      ok = sweeps >= 0;
#pragma unroll
      for (int c = 0; c < PP; ++c) Q[c] = sel4(Vr, ord[c]);
      gap = INFINITY;
      if constexpr (PP < 4) gap = sel4(lam, ord[PP]) - sel4(lam, ord[PP - 1]);
    }
  }
  gap /= a.scale;
  const bool write = active && l == 0;
  if (write) {
    a.gap[k] = gap;
    if (!ok) report(a.status, ST_ENOCONV, k, 0.0);
    if (!(gap > a.gap_tol)) report(a.status, ST_EGAP, k, gap);
  }
  if (a.op.nnz > 0) {
    if constexpr (PP % 2 == 0) {
      // projected spin operator restricted to the occupied space (Sec. IV)
      z64 sQ[PP], S[PP][PP];
#pragma unroll
      for (int c = 0; c < PP; ++c) sQ[c] = z64(0.0, 0.0);
      for (int q = 0; q < a.op.nnz; ++q) {
        const int col = a.op.col[q];
        const z64 v = a.op.row[q] == l ? a.op.val[q] : z64(0.0, 0.0);
#pragma unroll
        for (int c = 0; c < PP; ++c) cfma(sQ[c], v, shfl_z(Q[c], base + col));
      }
      quad_gram<PP>(Q, sQ, S, l, base);
      z64 v[PP][PP / 2];
      tiny_sector_columns<PP>(a, k, S, write, v);
      if (!active) return;
      z64* out = a.U + k * 4LL * (PP / 2) + l * (PP / 2);
#pragma unroll
      for (int c = 0; c < PP / 2; ++c) {
        z64 acc(0.0, 0.0);
#pragma unroll
        for (int q = 0; q < PP; ++q) cfma(acc, Q[q], v[q][c]);
        out[c] = acc;
      }
    }
    return;
  }
  if (!active) return;
  z64* out = a.U + k * 4LL * PP + l * PP;
#pragma unroll
  for (int c = 0; c < PP; ++c) out[c] = Q[c];
}

// n = 4 on large grids when H(k) is diagonal after a few rotations (the models with symmetry;
// four_band_rotations counts them): one thread per k-point, FP64 Jacobi, whose rotations of
// zero entries are skipped.  There the sweeps take fewer FP64 instructions than the refined
// solve, 20 rotations take twice as many, and below ~13 000 points four lanes per k-point finish
// before one thread's chain does.  States kernel, one thread / four lanes, us:
//   BBH (5 rotations)       9000 points 61 / 43, 18 000 65 / 78, 90 000 264 / 344, 230 400 635 / 866
//   spin-Hall (2), spin     9000 49 / 51, 18 000 53 / 92, 90 000 192 / 412, 230 400 463 / 1038
//   Eq. 9 (5)               18 000 72 / 82, 230 400 676 / 926
//   BBH + diagonal (22)     18 000 184 / 82, 230 400 1830 / 892 (as any other pattern of 8 to 16
//                           entries that does not end early)
constexpr int FOUR_THREADS = 32;

template <int PP>
__device__ __forceinline__ void states_four(const StatesArgs& a, int use_tab) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int eb[16], ee[16];
  const int tid = threadIdx.x, bd = blockDim.x;
  const TinySmem T = tiny_tables<4>(a, smem, bd, use_tab != 0, eb, ee);
  const long long k = (long long)blockIdx.x * bd + tid;
  if (k >= a.K) return;
  tiny_phases(a, T, k, tid, bd, use_tab != 0, 0, 1);
  z64 A[4][4], V[4][4], Vs[4][4];
  double lam[4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = r; c < 4; ++c) {
      A[r][c] = tiny_entry(T, eb[4 * r + c], ee[4 * r + c], tid, bd);
      if (r == c)
        A[r][r].im = 0.0;
      else
        A[c][r] = conj(A[r][c]);
    }
  const bool ok = jac_serial<4, double>(A, V, a.max_sweeps) >= 0;
  sort_eig<4, double>(A, V, Vs, lam);
  double gap = INFINITY;
  if constexpr (PP < 4) gap = lam[PP] - lam[PP - 1];
  a.gap[k] = gap;
  if (!ok) report(a.status, ST_ENOCONV, k, 0.0);
  if (!(gap > a.gap_tol)) report(a.status, ST_EGAP, k, gap);
  if (a.op.nnz > 0) {
    if constexpr (PP % 2 == 0) {
      // projected spin operator restricted to the occupied space (Sec. IV)
      z64 S[PP][PP];
#pragma unroll
      for (int x = 0; x < PP; ++x)
#pragma unroll
        for (int y = 0; y < PP; ++y) S[x][y] = z64(0.0, 0.0);
      for (int q = 0; q < a.op.nnz; ++q) {
        const int row = a.op.row[q], col = a.op.col[q];
        const z64 v = a.op.val[q];
        z64 qa[PP], qb[PP];
#pragma unroll
        for (int c = 0; c < PP; ++c) {
          qa[c] = qb[c] = z64(0.0, 0.0);
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            if (r == row) qa[c] = Vs[r][c];
            if (r == col) qb[c] = Vs[r][c];
          }
          qb[c] = v * qb[c];
        }
#pragma unroll
        for (int x = 0; x < PP; ++x)
#pragma unroll
          for (int y = 0; y < PP; ++y) cfma_conj(S[x][y], qa[x], qb[y]);
      }
#pragma unroll
      for (int x = 0; x < PP; ++x) {
        S[x][x].im = 0.0;
#pragma unroll
        for (int y = x + 1; y < PP; ++y) {
          S[x][y] = 0.5 * (S[x][y] + conj(S[y][x]));
          S[y][x] = conj(S[x][y]);
        }
      }
      z64 v[PP][PP / 2];
      tiny_sector_columns<PP>(a, k, S, true, v);
      z64* out = a.U + k * 4LL * (PP / 2);
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < PP / 2; ++c) {
          z64 acc(0.0, 0.0);
#pragma unroll
          for (int q = 0; q < PP; ++q) cfma(acc, Vs[r][q], v[q][c]);
          out[r * (PP / 2) + c] = acc;
        }
    }
    return;
  }
  z64* out = a.U + k * 4LL * PP;
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < PP; ++c) out[r * PP + c] = Vs[r][c];
}

template <int PP>
__global__ void __launch_bounds__(FOUR_THREADS) k_states_four(StatesArgs a, int use_tab) {
  states_four<PP>(a, use_tab);
}
template <int PP>
__global__ void __launch_bounds__(FOUR_THREADS)
    k_states_four_inl(StatesArgs a, int use_tab, const char* dbase, const __grid_constant__ FusedPlan plan) {
  tiny_relocate(a, plan.bytes, dbase);
  states_four<PP>(a, use_tab);
}

template <int PP>
__global__ void __launch_bounds__(TINY_THREADS) k_states_two(StatesArgs a, int use_tab) {
  states_two<PP>(a, use_tab);
}
template <int PP>
__global__ void __launch_bounds__(TINY_THREADS)
    k_states_two_inl(StatesArgs a, int use_tab, const char* dbase, const __grid_constant__ FusedPlan plan) {
  tiny_relocate(a, plan.bytes, dbase);
  states_two<PP>(a, use_tab);
}
template <int PP>
__global__ void __launch_bounds__(QUAD_THREADS) k_states_quad(StatesArgs a, int use_tab) {
  states_quad<PP>(a, use_tab);
}
template <int PP>
__global__ void __launch_bounds__(QUAD_THREADS)
    k_states_quad_inl(StatesArgs a, int use_tab, const char* dbase, const __grid_constant__ FusedPlan plan) {
  tiny_relocate(a, plan.bytes, dbase);
  states_quad<PP>(a, use_tab);
}

// ---------------------------------------------------------------------------
// Mixed precision, four lanes per k-point (n = 4, p = 2, no spin split), with every step on
// the FP32 pipe: GB300 issues FP32 about 70x faster than FP64.  Lane l of a group of four
// consecutive lanes holds row l of H(k) and of the eigenvector matrix (quad.cuh).
//  - Bloch phases and H(k) in double-float (two-level phase tables, exact products
//    of the double-float hopping amplitudes with the phases);
//  - FP32 Jacobi on the float part of H, made exactly Hermitian;
//  - one Newton correction of the occupied block Q in the FP32 eigenbasis, with the
//    residual R = H Q - Q rho in double-float: for each unoccupied FP32 vector z_a,
//    Q_c += z_a (z_a^dag R_c) / (rho_c - lam_a), rho_c = q_c^dag H q_c;
//  - one second-order Lowdin step with the Gram matrix in double-float;
//  - the gap from double-float Ritz values of the two FP32 pairs, to second order in what
//    they lack of orthonormality and of convergence (60 x 3840 points: at most 2.7e-13 off).
// The occupied block leaves as complex double-float (hi, lo per part, 16 bytes like
// a complex128), accurate to about 1e-13, for the double-float loop kernels.
// ---------------------------------------------------------------------------
size_t quad_df_smem(int nR, int N, int Nt) {
  const TabShape tN = tab_shape_split(N), tT = tab_shape_split(Nt);
  return (size_t(nR) * (QUAD_THREADS / 4) + tN.B + tN.H + tT.B + tT.H + nR) * sizeof(cdf) +
         3 * size_t(nR) * sizeof(int);
}

template <int PP>
__global__ void __launch_bounds__(QUAD_THREADS) k_states_quad_df(StatesArgs a) {
  static_assert(PP == 2, "the double-float four-lane kernel serves two occupied bands");
  extern __shared__ __align__(16) unsigned char smem[];
  const DevModel& md = a.model;
  const int tid = threadIdx.x, nR = md.n_R;
  const int N = a.plane.N, Nt = a.plane.N_t;
  const TabShape tN = tab_shape_split(N), tT = tab_shape_split(Nt);
  constexpr int KPB = QUAD_THREADS / 4;
  cdf* cache = reinterpret_cast<cdf*>(smem);   // nR x KPB
  cdf* tabN = cache + nR * KPB;
  cdf* tabNt = tabN + tN.B + tN.H;
  cdf* oph = tabNt + tT.B + tT.H;
  int* lR = reinterpret_cast<int*>(oph + nR);
  int* tR = lR + nR;
  int* sR = tR + nR;
  fill_tab_df(tabN, tabN + tN.B, N, tN);
  fill_tab_df(tabNt, tabNt + tT.B, Nt, tT);
  for (int r = tid; r < nR; r += blockDim.x) {
    const int* Rv = md.Rv + 3 * r;
    double x = 0.0;
    int lq = 0, tq = 0, sq = 0;
    for (int dd = 0; dd < 3; ++dd) {
      x += a.plane.origin[dd] * double(Rv[dd]);
      lq += int(a.plane.loop_dir[dd]) * Rv[dd];
      tq += int(a.plane.trans_dir[dd]) * Rv[dd];
      sq += a.plane.sweep[dd] * Rv[dd];
    }
    double sn, cs;
    sincospi(2.0 * x, &sn, &cs);
    oph[r] = cdf_from(z64(cs, sn));
    lR[r] = lq;
    tR[r] = tq;
    sR[r] = sq;
  }
  __syncthreads();
  const int l = tid & 3, kl = tid >> 2, base = (tid & 31) & ~3;
  const long long kraw = (long long)blockIdx.x * KPB + kl;
  const bool active = kraw < a.K;
  const long long k = active ? kraw : a.K - 1;  // idle groups recompute the last k-point
  const int i = int(k / N), j = int(k - (long long)i * N);
  for (int r = l; r < nR; r += 4) {
    const int mN = pmod((long long)j * lR[r], N), mT = pmod(plane_row_index(a.plane, i, tR[r], sR[r]), Nt);
    cache[r * KPB + kl] = oph[r] * tab_at_df(tabN, tabN + tN.B, tN, mN) *
                          tab_at_df(tabNt, tabNt + tT.B, tT, mT);
  }
  __syncwarp();
  // row l of H(k) in double-float
  cdf Hr[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) Hr[c] = cdf_zero();
  for (int e = a.row_ptr[l]; e < a.row_ptr[l + 1]; ++e) {
    cdf acc = cdf_zero();
    for (int h = md.ent_start[e]; h < md.ent_start[e + 1]; ++h) {
      const float* t4 = md.hop_tdf + 4 * h;
      cfma(acc, cdf(df(t4[0], t4[1]), df(t4[2], t4[3])), cache[md.hop_r[h] * KPB + kl]);
    }
    const int col = md.ent_col[e];
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (c == col) Hr[c] = acc;
  }
  cdf Qf[PP];
  double gap;
  const int sweeps = quad_df_occupied(Hr, l, base, a.max_sweeps, Qf[0], Qf[1], gap);
  if (!active) return;
  cdf* out = reinterpret_cast<cdf*>(a.U) + k * 4LL * PP + l * PP;
#pragma unroll
  for (int c = 0; c < PP; ++c) out[c] = Qf[c];
  if (l == 0) {
    a.gap[k] = gap;
    if (sweeps < 0) report(a.status, ST_ENOCONV, k, 0.0);
    if (!(gap > a.gap_tol)) report(a.status, ST_EGAP, k, gap);
  }
}

template <int PP>
cudaError_t quad_df_launch(const StatesArgs& a, size_t smem, cudaStream_t s) {
  static size_t cached = 0;
  cudaError_t e = set_smem_once(k_states_quad_df<PP>, smem, cached);
  if (e != cudaSuccess) return e;
  const long long blocks = (a.K + QUAD_THREADS / 4 - 1) / (QUAD_THREADS / 4);
  k_states_quad_df<PP><<<int(blocks), QUAD_THREADS, smem, s>>>(a);
  return cudaGetLastError();
}

template <int PP>
cudaError_t quad_launch(const StatesArgs& a, bool use_tab, TabShape tN, TabShape tT, cudaStream_t s,
                        const FusedPlan* plan, const char* dbase) {
  constexpr int KPB = QUAD_THREADS / 4;
  cudaError_t e;
  if (a.rotations > 0 && a.rotations <= FOUR_MAX_ROT && a.K > FOUR_MIN_K) {
    const size_t sm = tiny_smem_bytes(a.model.n_R, a.model.n_hop, FOUR_THREADS, use_tab, tN, tT);
    const int grid = int((a.K + FOUR_THREADS - 1) / FOUR_THREADS);
    if (plan) {
      static size_t cached_fi = 0;
      if ((e = set_smem_once(k_states_four_inl<PP>, sm, cached_fi)) != cudaSuccess) return e;
      k_states_four_inl<PP><<<grid, FOUR_THREADS, sm, s>>>(a, use_tab, dbase, *plan);
    } else {
      static size_t cached_f = 0;
      if ((e = set_smem_once(k_states_four<PP>, sm, cached_f)) != cudaSuccess) return e;
      k_states_four<PP><<<grid, FOUR_THREADS, sm, s>>>(a, use_tab);
    }
    return cudaGetLastError();
  }
  const size_t smem = tiny_smem_bytes(a.model.n_R, a.model.n_hop, KPB, use_tab, tN, tT);
  if (plan) {
    static size_t cached_i = 0;
    if ((e = set_smem_once(k_states_quad_inl<PP>, smem, cached_i)) != cudaSuccess) return e;
    k_states_quad_inl<PP><<<int((a.K + KPB - 1) / KPB), QUAD_THREADS, smem, s>>>(a, use_tab, dbase, *plan);
    return cudaGetLastError();
  }
  static size_t cached = 0;
  e = set_smem_once(k_states_quad<PP>, smem, cached);
  if (e != cudaSuccess) return e;
  k_states_quad<PP><<<int((a.K + KPB - 1) / KPB), QUAD_THREADS, smem, s>>>(a, use_tab);
  return cudaGetLastError();
}

template <int PP>
cudaError_t two_launch(const StatesArgs& a, bool use_tab, TabShape tN, TabShape tT, cudaStream_t s,
                        const FusedPlan* plan, const char* dbase) {
  const size_t smem = tiny_smem_bytes(a.model.n_R, a.model.n_hop, TINY_THREADS, use_tab, tN, tT);
  cudaError_t e;
  if (plan) {
    static size_t cached_i = 0;
    if ((e = set_smem_once(k_states_two_inl<PP>, smem, cached_i)) != cudaSuccess) return e;
    k_states_two_inl<PP><<<int((a.K + TINY_THREADS - 1) / TINY_THREADS), TINY_THREADS, smem, s>>>(a, use_tab, dbase, *plan);
    return cudaGetLastError();
  }
  static size_t cached = 0;
  e = set_smem_once(k_states_two<PP>, smem, cached);
  if (e != cudaSuccess) return e;
  k_states_two<PP><<<int((a.K + TINY_THREADS - 1) / TINY_THREADS), TINY_THREADS, smem, s>>>(a, use_tab);
  return cudaGetLastError();
}

}  // namespace

// The double-float four-lane kernel applies: mixed precision, n = 4, p = 2, no spin split,
// an integer plane (phase tables), at most TINY_R_MAX translations.
bool states_df_eligible(const StatesArgs& a, int p_out) {
  if (!a.mixed || a.f != nullptr || a.op.nnz > 0 || a.model.n != 4 || a.p != 2 ||
      p_out != a.p || a.model.n_R > TINY_R_MAX || a.K <= 0 || !a.row_ptr)
    return false;
  for (int d = 0; d < 3; ++d)
    if (a.plane.trans_dir[d] != double((long long)a.plane.trans_dir[d])) return false;
  return quad_df_smem(a.model.n_R, a.plane.N, a.plane.N_t) <= 48 * 1024;
}

bool tiny_takes(const StatesArgs& a, int p_out) {
  const int n = a.model.n, p = a.p;
  if (!(n == 2 || n == 4) || p < 1 || p > n || a.model.n_R > TINY_R_MAX || a.K <= 0) return false;
  return !(a.op.nnz > 0 && (p % 2 || p_out != p / 2));
}

bool states_plan_inline(const StatesArgs& a, int p_out) { return !a.want_df && tiny_takes(a, p_out); }

// Few-band path: n in {2, 4}, at most TINY_R_MAX distinct translations.  Sets
// *handled = false (and launches nothing) when the problem is outside it.
cudaError_t launch_states_tiny(const StatesArgs& a, int p_out, cudaStream_t s, bool* handled, const void* plan_host,
                               size_t plan_bytes, const void* plan_dev) {
  *handled = false;
  const int n = a.model.n, p = a.p;
  if (!tiny_takes(a, p_out)) return plan_host ? cudaErrorInvalidValue : cudaSuccess;
  if (plan_host && (a.want_df || plan_bytes > sizeof(FusedPlan))) return cudaErrorInvalidValue;
  FusedPlan plan;  // the kernel parameter (copied at launch)
  const FusedPlan* fp = nullptr;
  const char* dbase = static_cast<const char*>(plan_dev);
  if (plan_host) {
    std::memcpy(plan.bytes, plan_host, plan_bytes);
    std::memset(plan.bytes + plan_bytes, 0, sizeof(plan.bytes) - plan_bytes);
    fp = &plan;
  }
  const int N = a.plane.N, Nt = a.plane.N_t;
  bool integer_plane = a.f == nullptr;
  for (int d = 0; d < 3; ++d)
    integer_plane = integer_plane && a.plane.trans_dir[d] == double((long long)a.plane.trans_dir[d]);
  const TabShape tN = tab_shape(N), tT = tab_shape(Nt);
  const size_t tab = size_t(tN.B) + tN.H + tT.B + tT.H;
  const bool use_tab = integer_plane && tab <= 4096;
  *handled = true;
  if (a.want_df)  // the caller checked states_df_eligible()
    return quad_df_launch<2>(a, quad_df_smem(a.model.n_R, N, Nt), s);
  if (n == 2) return p == 1 ? two_launch<1>(a, use_tab, tN, tT, s, fp, dbase) : two_launch<2>(a, use_tab, tN, tT, s, fp, dbase);
  switch (p) {
    case 1: return quad_launch<1>(a, use_tab, tN, tT, s, fp, dbase);
    case 2: return quad_launch<2>(a, use_tab, tN, tT, s, fp, dbase);
    case 3: return quad_launch<3>(a, use_tab, tN, tT, s, fp, dbase);
    default: return quad_launch<4>(a, use_tab, tN, tT, s, fp, dbase);
  }
}

}  // namespace bw
