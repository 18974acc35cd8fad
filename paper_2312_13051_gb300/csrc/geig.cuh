// Block-wide eigensolver for a general complex matrix in shared memory (FP64).
//
// The Wilson matrix of Eq. 2 is a product of raw overlaps and is not unitary, so
// its eigenvalues need a general (non-Hermitian) solver: Householder reduction to
// upper Hessenberg form, then implicit QR sweeps with Givens rotations and deflation on
// small subdiagonals, several sweeps chasing each other through the matrix two rows apart,
// with the eigenvalues of the trailing block as their shifts.  With vectors
// requested the rotations are applied to whole rows/columns, leaving the Schur
// form T = Z^dagger W Z; right eigenvectors are x = Z y with T y = lambda y solved
// by back substitution.
#pragma once

#include "common.cuh"

namespace bw {

// Sweeps in flight.  A rotation is a chain of ~20 dependent FP64 operations (64 clocks each
// on GB300) and three block barriers, whatever the number of entries it moves, so the sweeps
// of several shifts share the steps: NB sweeps over an active block of s rows take
// s + 2 NB steps instead of NB s.  Measured (one CTA per loop, product included; one sweep at a
// time, now): p = 64 FP64, 27 loops, 32.4, 17.0 ms; p = 32 FP64, 17 loops, 5.5, 3.0 ms; p = 12
// with vectors, 31 loops, 1.56, 0.81 ms.  A step at p = 64 takes ~7000 clocks: 2100 the rotations,
// the rest FP64 throughput.
constexpr int GEIG_NB = 8;
constexpr int GEIG_STALL = 30;  // rounds without a deflation after which the product test decides too

struct GeigShared {
  double c[GEIG_NB];    // Givens of each sweep: G = [[c, s], [-conj(s), c]], c real
  z64 s[GEIG_NB];
  z64 shift[GEIG_NB];        // of each sweep
  c32 low[GEIG_NB];          // the same in FP32, scaled (shift selection)
  c32 B[GEIG_NB * GEIG_NB];  // trailing block
  z64 mu;
  int l, hi, nb, active, fail;
};

__device__ __forceinline__ double zabs(z64 a) { return hypot(a.re, a.im); }

// Givens G with G [x; y] = [r; 0], c real >= 0: c = |x| / r, s = (x / |x|) conj(y) / r,
// r = sqrt(|x|^2 + |y|^2), from two reciprocal square roots (the entries of the
// Wilson matrices are O(1), far from the range where the squares over- or
// underflow; a square that underflows makes the rotation swap the two rows, still
// unitary, and the entry it leaves behind is set to zero by the caller).
__device__ __forceinline__ void givens(z64 x, z64 y, double& c, z64& s) {
  const double ax2 = abs2(x), ay2 = abs2(y);
  if (ay2 == 0.0) {
    c = 1.0;
    s = z64(0.0, 0.0);
    return;
  }
  if (ax2 == 0.0) {
    c = 0.0;
    const double iy = rsqrt(ay2);
    s = z64(y.re * iy, -y.im * iy);  // conj(y)/|y|
    return;
  }
  const double ir = rsqrt(ax2 + ay2), iax = rsqrt(ax2);
  c = ax2 * iax * ir;
  const z64 ux(x.re * iax, x.im * iax);
  s = ir * (ux * conj(y));
}

// Whether the subdiagonal entry H[l][l-1] is negligible: against the neighbouring
// diagonal entries, or by the product test of Ahues and Tisseur (its product with the
// superdiagonal small against the local separation of the diagonal entries).
// Magnitudes are |re| + |im| (within a factor sqrt(2) of the modulus, a hypot each otherwise).
// The product test can let go of entries far above rounding where the superdiagonal one is
// small.  That is right for the 2 x 2 block, but several sweeps at once leave many such entries
// inside a matrix that has not converged, where what is dropped couples to everything right of
// the superdiagonal: phases of weakly coupled bands lost two digits (p = 32 to 80, FP64: up to
// 8e-13 rad from FP64, without it 1e-14).  So those sweeps use it for entries up to 64 roundings
// (`product` false), what a block of equal eigenvalues, whose off-diagonal entries are rounding
// themselves, needs in order to fall apart; any entry only after GEIG_STALL rounds without a
// deflation.  The cluster solver, one sweep at a time, uses it for any entry.
__device__ __forceinline__ double zabs1(z64 a) { return fabs(a.re) + fabs(a.im); }

__device__ __forceinline__ bool geig_negligible_v(z64 h11, z64 h12, z64 h21, z64 h22, double eps, bool product) {
  const double sub = zabs1(h21);
  const double dia = zabs1(h22) + zabs1(h11);
  bool small = sub <= eps * dia || sub < 1e-300;
  if (!small && sub <= (product ? 1.0 : 64.0 * eps) * dia) {
    const double x = zabs1(h12);
    const double ab = fmax(sub, x), ba = fmin(sub, x);
    const double y = zabs1(h11 - h22);
    const double aa = fmax(zabs1(h22), y), bb = fmin(zabs1(h22), y);
    const double sc = aa + ab;
    small = ba * (ab / sc) <= fmax(1e-300, eps * (bb * (aa / sc)));
  }
  return small;
}

__device__ __forceinline__ bool geig_negligible(const z64* H, int ld, int l, double eps, bool product) {
  return geig_negligible_v(H[(l - 1) * ld + l - 1], H[(l - 1) * ld + l], H[l * ld + l - 1],
                           H[l * ld + l], eps, product);
}

// Shift of a QR sweep from the trailing 2 x 2 [[a, b], [c, d]] of the active window:
// its eigenvalue closest to d (Wilkinson); every 12th sweep without a deflation the
// exceptional shift d + 0.75 (|c| + sub2), sub2 = |H[hi-1][hi-2]| (0 when hi < 2).
__device__ __forceinline__ z64 geig_shift(z64 a, z64 b, z64 c, z64 d, int iter, double sub2) {
  if (iter > 0 && iter % 12 == 0) return d + z64(0.75 * (zabs(c) + sub2), 0.0);
  const z64 half = 0.5 * (a - d);
  const z64 disc = half * half + b * c;
  // complex sqrt
  const double r = zabs(disc);
  const double sr = sqrt(0.5 * (r + fabs(disc.re)));
  z64 sq;
  if (sr == 0.0) {
    sq = z64(0.0, 0.0);
  } else if (disc.re >= 0.0) {
    sq = z64(sr, disc.im / (2.0 * sr));
  } else {
    sq = z64(fabs(disc.im) / (2.0 * sr), disc.im >= 0.0 ? sr : -sr);
  }
  // mu = d + half -/+ sq, the one closer to d
  const z64 m1 = d + half - sq, m2 = d + half + sq;
  return (abs2(m1 - d) <= abs2(m2 - d)) ? m1 : m2;
}

// 2^-e with 2^e <= m < 2^(e+1), from the exponent bits (m finite, below 2^127; subnormal m and
// zero give 2^127): a scaling without rounding that brings m into [1, 2).
__device__ __forceinline__ float geig_unit(float m) {
  return __int_as_float(0x7f000000 - (__float_as_int(m) & 0x7f800000));
}
__device__ __forceinline__ float geig_max(c32 a, c32 b) {
  return fmaxf(fmaxf(fabsf(a.re), fabsf(a.im)), fmaxf(fabsf(b.re), fabsf(b.im)));
}
__device__ __forceinline__ float geig_abs1(c32 a) { return fabsf(a.re) + fabsf(a.im); }

// Shifts of nb simultaneous sweeps: the eigenvalues of the trailing nb x nb block B (FP32,
// Hessenberg, entries at most 2) of the active window by single-shift QR (a shift decides how
// fast the sweeps converge, not what they converge to), in the order in which they separate
// from the bottom.  At its cap of sweeps the diagonal entries left over serve.  The block of
// a nearly singular Wilson matrix spans the whole FP32 range, so nothing below squares an
// entry or takes the reciprocal of one without scaling it by a power of two first: every
// shift is finite.  One warp calls it, all lanes; nb <= 32.
__device__ __forceinline__ void geig_block_shifts(c32* B, int nb, c32* shift) {
  const int lane = threadIdx.x & 31;
  int top = nb - 1, out = 0;
  for (int it = 0; it < 8 * GEIG_NB && top > 0; ++it) {
    // split point: the largest l whose subdiagonal entry is negligible
    const bool small = lane >= 1 && lane <= top &&
                       geig_abs1(B[lane * nb + lane - 1]) <=
                           1e-6f * (geig_abs1(B[lane * nb + lane]) + geig_abs1(B[(lane - 1) * nb + lane - 1]));
    const unsigned m = __ballot_sync(0xffffffffu, small);
    const int l = m ? 31 - __clz(m) : 0;
    if (l == top) {
      if (lane == 0) shift[out] = B[top * nb + top];
      ++out;
      --top;
      continue;
    }
    // Wilkinson shift: the eigenvalue of the last 2 x 2 block [[a, b], [c, d]] closest to d,
    // d - b c / (g +- sqrt(g^2 + b c)) with g = (a - d) / 2 and the larger denominator
    c32 a = B[(top - 1) * nb + top - 1], b = B[(top - 1) * nb + top], c = B[top * nb + top - 1], d = B[top * nb + top];
    const float u2 = geig_unit(fmaxf(geig_max(a, b), geig_max(c, d)));
    a = u2 * a;
    b = u2 * b;
    c = u2 * c;
    const c32 bc = b * c, g = 0.5f * (a - u2 * d), q = g * g + bc;
    const float sr = sqrtf(0.5f * (hypotf(q.re, q.im) + fabsf(q.re)));
    c32 sq(0.f, 0.f);
    if (sr > 0.f)
      sq = q.re >= 0.f ? c32(sr, 0.5f * q.im / sr) : c32(0.5f * fabsf(q.im) / sr, copysignf(sr, q.im));
    if (g.re * sq.re + g.im * sq.im < 0.f) sq = -sq;
    const c32 den = g + sq;
    const float d2 = abs2(den);
    const c32 mu = d2 > 1e-30f ? d - (1.f / u2) * ((1.f / d2) * (bc * conj(den))) : d;
    for (int k = l; k < top; ++k) {
      c32 x = k == l ? B[l * nb + l] - mu : B[k * nb + k - 1];
      c32 y = k == l ? B[(l + 1) * nb + l] : B[(k + 1) * nb + k - 1];
      const float m1 = geig_max(x, y);
      float cr = 1.f;
      c32 s(0.f, 0.f);
      if (m1 > 0.f) {
        const float u1 = geig_unit(m1);
        x = u1 * x;
        y = u1 * y;
        const float ax2 = abs2(x), ir = rsqrtf(ax2 + abs2(y));
        if (ax2 > 1e-30f) {
          const float iax = rsqrtf(ax2);
          cr = ax2 * iax * ir;
          s = (iax * x) * conj(ir * y);
        } else {
          cr = 0.f;
          s = ir * conj(y);
        }
      }
      __syncwarp();
      const int cb = k > l ? k - 1 : l;
      if (lane >= cb && lane <= top) {
        const c32 u = B[k * nb + lane], v = B[(k + 1) * nb + lane];
        B[k * nb + lane] = cr * u + s * v;
        B[(k + 1) * nb + lane] = cr * v - conj(s) * u;
      }
      __syncwarp();
      if (lane >= l && lane <= min(k + 2, top)) {
        const c32 u = B[lane * nb + k], v = B[lane * nb + k + 1];
        B[lane * nb + k] = cr * u + v * conj(s);
        B[lane * nb + k + 1] = cr * v - u * s;
      }
      __syncwarp();
      if (lane == 0 && k > l) B[(k + 1) * nb + k - 1] = c32(0.f, 0.f);
      __syncwarp();
    }
  }
  if (lane <= top) shift[out + lane] = B[(top - lane) * nb + top - lane];
  __syncwarp();
}

// The same from the trailing block of the matrix itself (rows hi - nb + 1 .. hi): scaled by a
// power of two to FP32, its entries below 2; returns the power that the shifts are to be
// multiplied by, or 0 when a shift is not finite (the matrix itself is not).  Shifts that FP32
// does not tell apart (an eigenvalue of W that many bands share) are kept once: nb becomes
// the number kept.
__device__ __forceinline__ double geig_shifts(const z64* H, int ld, int hi, int& nb, c32* B, c32* shift) {
  const int lane = threadIdx.x & 31, h0 = hi - nb + 1;
  unsigned top = 0;  // leading word of the largest magnitude
  for (int e = lane; e < nb * nb; e += 32) {
    const int r = e / nb, c = e - r * nb;
    if (r > c + 1) continue;
    const z64 v = H[(h0 + r) * ld + h0 + c];
    top = max(top, max(unsigned(__double2hiint(fabs(v.re))), unsigned(__double2hiint(fabs(v.im)))));
  }
  top = __reduce_max_sync(0xffffffffu, top);
  const int ex = min(max(int(top >> 20), 1), 2045);
  const double down = __hiloint2double((2046 - ex) << 20, 0);
  for (int e = lane; e < nb * nb; e += 32) {
    const int r = e / nb, c = e - r * nb;
    B[e] = r <= c + 1 ? ccast<float>(down * H[(h0 + r) * ld + h0 + c]) : c32(0.f, 0.f);
  }
  __syncwarp();
  geig_block_shifts(B, nb, shift);
  const c32 s = lane < nb ? shift[lane] : c32(0.f, 0.f);
  const bool ok = isfinite(s.re) && isfinite(s.im);
  bool keep = lane < nb;
  for (int j = 0; j + 1 < nb; ++j) {
    const c32 o(__shfl_sync(0xffffffffu, s.re, j), __shfl_sync(0xffffffffu, s.im, j));
    if (j < lane && geig_abs1(s - o) < 4e-6f) keep = false;
  }
  const unsigned m = __ballot_sync(0xffffffffu, keep);
  __syncwarp();
  if (keep) shift[__popc(m & ((1u << lane) - 1u))] = s;
  nb = __popc(m);
  __syncwarp();
  return __all_sync(0xffffffffu, ok) ? __hiloint2double(ex << 20, 0) : 0.0;
}

// Largest l in [1, hi] whose subdiagonal entry is negligible, or 0: the first warp
// tests 32 subdiagonals at a time from hi down.  Every lane of the warp calls it.
__device__ __forceinline__ int geig_split_point(const z64* H, int ld, int hi, double eps, bool product) {
  const int lane = threadIdx.x & 31;
  for (int base = hi; base >= 1; base -= 32) {
    const int l = base - lane;
    const bool f = l >= 1 && geig_negligible(H, ld, l, eps, product);
    const unsigned m = __ballot_sync(0xffffffffu, f);
    if (m) return base - (__ffs(m) - 1);
  }
  return 0;
}

// Eigen-decomposition of H (p x p, leading dimension ld), destroyed on output.
// lam[p] receives the eigenvalues.  With want_vec, Z (p x p) receives the right
// eigenvectors as unit-norm columns; vec scratch needs p z64.  Returns 0, or -1
// when the QR iteration cap (120 p + 120 rounds of sweeps) is reached.
__device__ inline int geig(z64* H, z64* Z, int p, int ld, bool want_vec, z64* lam, z64* vec,
                    GeigShared* sh) {
  const int tid = threadIdx.x, nt = blockDim.x;
  const double eps = 2.220446049250313e-16;
  if (want_vec)
    for (int e = tid; e < p * p; e += nt) {
      const int r = e / p, c = e - r * p;
      Z[r * ld + c] = z64(double(r == c), 0.0);
    }
  __syncthreads();
  // --- Householder reduction to Hessenberg form.  Column norms are block
  // reductions; the left update runs one thread per column and the right update one
  // warp per row, so that consecutive threads touch consecutive entries.
  __shared__ double hred[32];
  const int lane = tid & 31, warp = tid >> 5, nwarp = (nt + 31) >> 5;
  for (int c = 0; c + 2 < p; ++c) {
    double nrm2 = 0.0;
    for (int r = c + 1 + tid; r < p; r += nt) nrm2 += abs2(H[r * ld + c]);
    nrm2 = block_sum(nrm2, hred);
    const z64 x0 = H[(c + 1) * ld + c];
    const double tail = nrm2 - abs2(x0);
    if (!(tail > 0.0)) {
      __syncthreads();
      continue;
    }
    const double nx = sqrt(nrm2), ax0 = zabs(x0);
    const z64 ph = ax0 > 0.0 ? z64(x0.re / ax0, x0.im / ax0) : z64(1.0, 0.0);
    // v = x - alpha e1, alpha = -|x| ph: v_0 = ph (|x0| + |x|), |v|^2 = (|x0| + |x|)^2 + tail
    const double v0m = ax0 + nx, nv = 1.0 / sqrt(v0m * v0m + tail);
    for (int r = c + 1 + tid; r < p; r += nt)
      vec[r] = r == c + 1 ? z64(nv * v0m * ph.re, nv * v0m * ph.im) : nv * H[r * ld + c];
    if (tid == 0) sh->mu = -nx * ph;
    __syncthreads();
    // left: H <- (I - 2 v v^dagger) H on rows c+1.., columns c+1.. (column c is set below);
    // a warp takes eight columns, four lanes per column share its rows
    for (int cb = c + 1 + 8 * warp; cb < p; cb += 8 * nwarp) {
      const int col = cb + (lane & 7), r0 = c + 1 + (lane >> 3);
      z64 w(0.0, 0.0);
      if (col < p)
        for (int r = r0; r < p; r += 4) cfma_conj(w, vec[r], H[r * ld + col]);
      for (int o = 8; o < 32; o <<= 1) {
        w.re += __shfl_xor_sync(0xffffffffu, w.re, o);
        w.im += __shfl_xor_sync(0xffffffffu, w.im, o);
      }
      w = 2.0 * w;
      if (col < p)
        for (int r = r0; r < p; r += 4) cfms(H[r * ld + col], vec[r], w);
    }
    __syncthreads();
    // right: H <- H (I - 2 v v^dagger) on columns c+1..; Z likewise
    for (int row = warp; row < p; row += nwarp) {
      z64* hr = H + row * ld;
      z64 w(0.0, 0.0);
      for (int k = c + 1 + lane; k < p; k += 32) cfma(w, hr[k], vec[k]);
      for (int o = 16; o > 0; o >>= 1) {
        w.re += __shfl_xor_sync(0xffffffffu, w.re, o);
        w.im += __shfl_xor_sync(0xffffffffu, w.im, o);
      }
      w = 2.0 * w;
      for (int k = c + 1 + lane; k < p; k += 32) cfms(hr[k], w, conj(vec[k]));
      if (want_vec) {
        z64* zr = Z + row * ld;
        z64 wz(0.0, 0.0);
        for (int k = c + 1 + lane; k < p; k += 32) cfma(wz, zr[k], vec[k]);
        for (int o = 16; o > 0; o >>= 1) {
          wz.re += __shfl_xor_sync(0xffffffffu, wz.re, o);
          wz.im += __shfl_xor_sync(0xffffffffu, wz.im, o);
        }
        wz = 2.0 * wz;
        for (int k = c + 1 + lane; k < p; k += 32) cfms(zr[k], wz, conj(vec[k]));
      }
    }
    __syncthreads();
    for (int r = c + 1 + tid; r < p; r += nt) H[r * ld + c] = r == c + 1 ? sh->mu : z64(0.0, 0.0);
    __syncthreads();
  }
  // --- shifted QR on the Hessenberg matrix
  if (tid == 0) {
    sh->hi = p - 1;
    sh->fail = 0;
  }
  __syncthreads();
  int iter = 0, total = 0;
  bool one = false;  // one sweep at a time from here on
  const int cap = 120 * p + 120;
  while (true) {
    if (tid < 32) {  // the first warp finds the active block and the shifts
      int hi = sh->hi, l = 0, nb = 0;
      while (hi >= 0) {
        if (hi == 0) {
          if (tid == 0) lam[0] = H[0];
          hi = -1;
          break;
        }
        l = geig_split_point(H, ld, hi, eps, one || iter >= GEIG_STALL);
        __syncwarp();
        if (tid == 0 && l > 0) H[l * ld + l - 1] = z64(0.0, 0.0);
        if (l == hi) {
          if (tid == 0) lam[hi] = H[hi * ld + hi];
          --hi;
          iter = 0;
          continue;
        }
        const int size = hi - l + 1;
        // one sweep on short blocks, and now and then when nothing deflates (exceptional
        // shifts); the last of several sweeps takes the 2 x 2 block's shift in FP64 as well: it
        // is the one that ends the convergence (p = 64, 27 loops: 10.5 -> 9.3 ms)
        nb = one || size < 6 || (iter > 0 && iter % 12 == 0) ? 1 : min(GEIG_NB, size / 3);
        if (nb > 1) {
          const int want = nb;
          const double up = geig_shifts(H, ld, hi, nb, sh->B, sh->low);
          one = 3 * nb <= want;  // eigenvalues shared by many bands: the block tells too little
          if (up > 0.0) {
            if (tid < nb) sh->shift[tid] = up * ccast<double>(sh->low[tid]);
          } else {
            nb = 1;
          }
        }
        __syncwarp();
        if (tid == 0) {
          sh->shift[nb - 1] =
              geig_shift(H[(hi - 1) * ld + hi - 1], H[(hi - 1) * ld + hi], H[hi * ld + hi - 1], H[hi * ld + hi],
                         iter, hi >= 2 ? zabs(H[(hi - 1) * ld + hi - 2]) : 0.0);
        }
        break;
      }
      ++iter;
      ++total;
      if (tid == 0) {
        sh->hi = hi;
        sh->l = l;
        sh->nb = nb;
        sh->active = nb > 0;
        if (total > cap) {
          sh->fail = 1;
          sh->active = 0;
        }
      }
    }
    __syncthreads();
    if (!sh->active) break;
    const int l = sh->l, hi = sh->hi, nb = sh->nb;
    const int col_end = want_vec ? p - 1 : hi;
    const int row_beg = want_vec ? 0 : l;
    // Sweep b is at row k_b = l + t - 2 b in step t.  The sweeps of a step act on disjoint
    // row pairs and disjoint column pairs, and left and right rotations commute, so all row
    // rotations and then all column rotations give what the sweeps give one after another.
    const int steps = hi - l + 2 * (nb - 1);
    const int ncb = (col_end - l) / 32 + 1, nrb = (hi - row_beg) / 32 + 1, nzb = want_vec ? (p - 1) / 32 + 1 : 0;
    for (int t = 0; t < steps; ++t) {
      if (tid < nb) {
        const int k = l + t - 2 * tid;
        if (k >= l && k < hi) {
          z64 x, y;
          if (k == l) {
            x = H[l * ld + l] - sh->shift[tid];
            y = H[(l + 1) * ld + l];
          } else {
            x = H[k * ld + k - 1];
            y = H[(k + 1) * ld + k - 1];
          }
          double c;
          z64 s;
          givens(x, y, c, s);
          sh->c[tid] = c;
          sh->s[tid] = s;
        }
      }
      __syncthreads();
      // rows k, k+1: [rk; rk1] <- G [rk; rk1], the annihilated entry set to zero
      for (int w = warp; w < nb * ncb; w += nwarp) {
        const int b = w / ncb, k = l + t - 2 * b, col = l + 32 * (w - b * ncb) + lane;
        if (k < l || k >= hi || col > col_end || col < k - 1) continue;
        const double c = sh->c[b];
        const z64 s = sh->s[b], x = H[k * ld + col], y = H[(k + 1) * ld + col];
        H[k * ld + col] = c * x + s * y;
        H[(k + 1) * ld + col] = k > l && col == k - 1 ? z64(0.0, 0.0) : c * y - conj(s) * x;
      }
      __syncthreads();
      // columns k, k+1: H <- H G^dagger; Z <- Z G^dagger
      for (int w = warp; w < nb * (nrb + nzb); w += nwarp) {
        const int b = w / (nrb + nzb), k = l + t - 2 * b;
        if (k < l || k >= hi) continue;
        int q = w - b * (nrb + nzb);
        const bool zr = q >= nrb;
        if (zr) q -= nrb;
        const int row = (zr ? 0 : row_beg) + 32 * q + lane;
        if (row > (zr ? p - 1 : min(k + 2, hi))) continue;
        z64* M = (zr ? Z : H) + row * ld;
        const double c = sh->c[b];
        const z64 s = sh->s[b], x = M[k], y = M[k + 1];
        M[k] = c * x + y * conj(s);
        M[k + 1] = c * y - x * s;
      }
      __syncthreads();
    }
  }
  const int fail = sh->fail;
  __syncthreads();
  if (fail) return -1;
  if (!want_vec) return 0;
  // --- right eigenvectors of the triangular T by back substitution; column k of
  // the result replaces column k of Z (T stays in H's upper triangle).
  double tn = 0.0;
  for (int e = tid; e < p * p; e += nt) {
    const int r = e / p, c = e - r * p;
    if (c >= r) tn = fmax(tn, zabs(H[r * ld + c]));
  }
  __shared__ double tmax[32];
  tn = -block_min(-tn, tmax);
  const double small = fmax(eps * tn, 1e-300);
  // One thread per eigenvector: y_k by back substitution, kept in row k left of the diagonal
  // (free below T), y_k[k] = 1.  (One thread for all of them, a division and a chain of sums
  // per entry, was a quarter of the solver at p = 12.)
  for (int k = tid; k < p; k += nt) {
    z64* y = H + k * ld;
    const z64 lk = H[k * ld + k];
    for (int r = k - 1; r >= 0; --r) {
      z64 acc = H[r * ld + k];
      for (int c = r + 1; c < k; ++c) cfma(acc, H[r * ld + c], y[c]);
      z64 den = H[r * ld + r] - lk;
      if (zabs(den) < small) den = z64(small, 0.0);
      const double dd = abs2(den);
      y[r] = z64(-(acc.re * den.re + acc.im * den.im) / dd, -(acc.im * den.re - acc.re * den.im) / dd);
    }
  }
  __syncthreads();
  // X = Z Y row by row, columns from the right: column k only uses columns <= k of the
  // original row
  for (int row = tid; row < p; row += nt) {
    z64* z = Z + row * ld;
    for (int k = p - 1; k >= 0; --k) {
      const z64* y = H + k * ld;
      z64 acc = z[k];
      for (int c = 0; c < k; ++c) cfma(acc, z[c], y[c]);
      z[k] = acc;
    }
  }
  __syncthreads();
  for (int k = warp; k < p; k += nwarp) {  // unit columns
    double s2 = 0.0;
    for (int r = lane; r < p; r += 32) s2 += abs2(Z[r * ld + k]);
    for (int o = 16; o > 0; o >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    const double inv = 1.0 / sqrt(s2);
    for (int r = lane; r < p; r += 32) Z[r * ld + k] = inv * Z[r * ld + k];
  }
  __syncthreads();
  return 0;
}

// Principal complex square root.
__device__ __forceinline__ z64 csqrt64(z64 z) {
  const double r = zabs(z);
  if (r == 0.0) return z64(0.0, 0.0);
  const double t = sqrt(0.5 * (r + fabs(z.re)));
  if (z.re >= 0.0) return z64(t, z.im / (2.0 * t));
  return z64(fabs(z.im) / (2.0 * t), z.im >= 0.0 ? t : -t);
}

// Closed-form eigen-decomposition of a 2 x 2 complex matrix H = [[a, b], [c, d]]
// (leading dimension ld), one thread: lam[0..2), and with Z the unit right
// eigenvectors as columns.  lambda = (a + d)/2 +- sqrt(((a - d)/2)^2 + b c); the
// root of larger magnitude comes from the formula and the other from
// det / lambda_1, which avoids cancellation.  Eigenvector of lambda: (b, lambda - a)
// or (lambda - d, c), whichever is longer (e_1, e_2 when H is a multiple of I).
__device__ inline void eig2_closed(const z64* H, int ld, z64* lam, z64* Z, bool want_vec) {
  const z64 a = H[0], b = H[1], c = H[ld], d = H[ld + 1];
  const z64 mid = 0.5 * (a + d), half = 0.5 * (a - d);
  const z64 sq = csqrt64(half * half + b * c);
  const z64 l1p = mid + sq, l1m = mid - sq;
  const z64 l1 = abs2(l1p) >= abs2(l1m) ? l1p : l1m;
  const z64 det = a * d - b * c;
  z64 l2;
  if (abs2(l1) > 0.0) {
    const double den = abs2(l1);
    l2 = z64((det.re * l1.re + det.im * l1.im) / den, (det.im * l1.re - det.re * l1.im) / den);
  } else {
    l2 = z64(0.0, 0.0);
  }
  lam[0] = l1;
  lam[1] = l2;
  if (!want_vec) return;
  for (int k = 0; k < 2; ++k) {
    const z64 l = lam[k];
    z64 v0 = b, v1 = l - a;
    const z64 w0 = l - d, w1 = c;
    if (abs2(w0) + abs2(w1) > abs2(v0) + abs2(v1)) {
      v0 = w0;
      v1 = w1;
    }
    double nv = abs2(v0) + abs2(v1);
    if (!(nv > 0.0)) {
      v0 = z64(k == 0 ? 1.0 : 0.0, 0.0);
      v1 = z64(k == 0 ? 0.0 : 1.0, 0.0);
      nv = 1.0;
    }
    const double inv = 1.0 / sqrt(nv);
    Z[0 * ld + k] = inv * v0;
    Z[1 * ld + k] = inv * v1;
  }
}

}  // namespace bw
