// Smallest right singular vector of the tile A-hat (the rows outside I_j) for
// the DIAF-S warp kernels, without a full SVD.  One warp per column, lane q
// owns column q of every k x k matrix.  In the working type S:
//
//   H = A-hat^* A-hat from A-hat's own rows and its inverse by symmetric
//     sweeps (no pivoting: H is positive definite), kept when the
//     column-scaled kappa = max_c sqrt(H_cc / pivot_c) is at most
//     smallest_kappa_max (its error is eps kappa^2 relative to that scaling);
//   inverse iteration until the Rayleigh quotient d settles to 1 %;
//   the inverse M of H - s I, s = d + tau, tau = 1.2e-5 ||H||_inf: by Sylvester's
//     law of inertia exactly one negative pivot proves that exactly one
//     eigenvalue lies below s, so an eigenvalue found below s is the smallest
//     and the next one is at least s away: the gap tests of the callers (the
//     1e-5 smax^2 hand-back, the 1e-6 smax DEGENERATE flag) cannot fire,
//     because ||H||_inf >= smax^2;
//   two corrections x <- x + dx, (H - d I) dx = -(H x - d x), with
//     (H - d I)^-1 = (M^-1 + (s - d) I)^-1 by two Neumann steps.
//
// Then the same corrections with the residual H x - d x taken from the FP64
// tile (A-hat^* (A-hat x)) until the predicted error is below kCorrectTol; each
// gains the working type's digits over ||H|| / gap (FP32: 5-6 digits on the
// stencil tiles, so two corrections).  Anything out of line -- a larger
// kappa, a pivot that is not a positive number, another inertia, an
// eigenvalue not below s, slow convergence, non-finite values -- returns
// false, and the caller runs the Householder QR and the Jacobi SVD.
//
// Why not the Jacobi: only one singular vector and the bound on the next
// singular value are needed, and a one-sided Jacobi pays about five sweeps of
// k^2 / 2 rotations of 6 k flops for them; the two inverses cost k^3 each and
// a correction 6 k^2, all of it independent multiply-adds.  (LDL^* factors
// with triangular solves have half the arithmetic, but every solve is a chain
// of 2 k dependent shuffles.)  Numeric pass before and after, on one GB300,
// with the Gram matrices and FP64 products over the rows' nonzeros: lognormal
// 64^3 (k = 25) 65.8 -> 16.3 ms, FP64 convection-diffusion 129^2 (k = 13)
// 11.3 -> 2.4 ms, complex Helmholtz 512^2 (k = 9) 13.3 -> 8.5 ms.
// What bounds it now is latency: three to four warps per scheduler on chains
// of shuffles and shared-memory reads.
#pragma once

#include "warp_la.cuh"

// A factor of the Gram matrix carries eps kappa^2.
template <class R> __device__ __forceinline__ constexpr R smallest_kappa_max() { return sizeof(R) == 4 ? R(30) : R(300); }
// Not for complex128: there the Jacobi stays.  Its W and V agree with this
// form's to 1e-14, but the residual at which a restarted GMRES stops moves by
// 1e-6 of itself with the last bits of W and V (Helmholtz 150^2, against a
// 64-bit restatement: 6.9e-7 with the Jacobi, 1.5e-6 with this form).
template <class S, int KMAX>
constexpr bool kSmallestFits = !(ScalarInfo<S>::cplx && sizeof(S) == 16);
constexpr int kInverseItMax = 16;
constexpr int kCorrectMax = 8;
// Predicted error after the last correction.  Less than 1e-14 gains nothing
// (errors of W, V and the applied vector against 64 bits stay the same at 1e-15
// and 1e-16), but columns whose corrections have reached rounding then count as
// not converging and go to the SVD (Helmholtz 512^2 11.2 -> 15.2 ms at 1e-15).
constexpr double kCorrectTol = 1e-14;

// (T^* z)_c of lane c in FP64 over the m tile rows; tiles of up to 16 columns
// split the rows between the half-warps.
template <class SD, int LDT, int KMAX>
__device__ __forceinline__ SD tile_adj_mul(const SD* Ts, const SD* zz, int m, int k, int lane) {
  SD g = sc_zero<SD>();
  if constexpr (KMAX <= 16) {
    const int c = lane & 15;
    if (c < k)
      for (int r = lane >> 4; r < m; r += 2) g = sc_cmadd(g, Ts[r + c * LDT], zz[r]);
    g += shfl_xor(g, 16);
  } else {
    if (lane < k)
      for (int r = 0; r < m; ++r) g = sc_cmadd(g, Ts[r + lane * LDT], zz[r]);
  }
  return g;
}

// x in the working type; what underflows there becomes its smallest number, not
// zero: the FP64 products go by the places that are not zero.
template <class S, class SD>
__device__ __forceinline__ S cast_keep(SD x) {
  if constexpr (std::is_same<S, SD>::value) {
    return x;
  } else if constexpr (ScalarInfo<SD>::cplx) {
    return {cast_keep<float>(x.re), cast_keep<float>(x.im)};
  } else {
    const float v = (float)x;
    return v == 0.0f && (top_word(x) | __double2loint(x)) != 0u ? __uint_as_float(1u) : v;
  }
}

// Copies the tile to the working type (rows in I_j as zeros when inI is given)
// and notes which columns each of the lane's rows (lane + 32u) has, all of
// them, I_j's too.
template <class S, class SD, int KMAX, int MMAX, int LDT>
__device__ __forceinline__ void copy_tile(const SD* Ts, const int32_t* inI, S* Tw, int m, int k, int lane,
                                          uint32_t (&rowmask)[MMAX / DIAF_WARP]) {
#pragma unroll
  for (int u = 0; u < MMAX / DIAF_WARP; ++u) {
    rowmask[u] = 0;
    const int r = lane + DIAF_WARP * u;
    if (r < m) {
      const bool out = inI && inI[r] >= 0;
      for (int c = 0; c < k; ++c) {
        const S v = cast_keep<S>(Ts[r + c * LDT]);
        if (sc_real(v) != RealOf<S>(0) || sc_imag(v) != RealOf<S>(0)) rowmask[u] |= 1u << c;
        Tw[r + c * LDT] = out ? sc_zero<S>() : v;
      }
    }
  }
  __syncwarp();
}

// H = W^* W (k x k, leading dimension KP; W's leading dimension LDT) and the
// rows with a nonzero in column `lane` (up to 16 columns: in column lane mod 16,
// the rows of the lane's half).  rowmask: a superset of the columns that the
// lane's rows have.  Tiles of up to 16 columns: a lane forms a column in
// registers, the half-warps alternate rows.  Wider ones, where the rows are
// short (a stencil's 7 of 25): lane q goes over its column's rows and each
// row's columns only, adding into its own column of H; m k steps per lane
// otherwise.
template <class S, int KMAX, int MMAX, int LDT, int KP>
__device__ __forceinline__ void tile_gram(const S* W, const uint32_t (&rowmask)[MMAX / DIAF_WARP], S* H, int m, int k,
                                          int lane, uint32_t (&colmask)[MMAX / DIAF_WARP]) {
  constexpr bool kHalf = KMAX <= 16;
  constexpr int NR = MMAX / DIAF_WARP;
  const int q = kHalf ? lane & 15 : lane;
  const bool own = q < k;
  if constexpr (!kHalf) {
    int steps = 0;
#pragma unroll
    for (int u = 0; u < NR; ++u) {
      colmask[u] = 0;
      for (int r = DIAF_WARP * u; r < m && r < DIAF_WARP * (u + 1); ++r) {  // row r's columns to their lanes
        const uint32_t b = __shfl_sync(DIAF_FULL, rowmask[u], r & 31);
        const bool has = own && (b >> lane & 1u) &&
                         (sc_real(W[r + q * LDT]) != RealOf<S>(0) || sc_imag(W[r + q * LDT]) != RealOf<S>(0));
        if (has) {
          colmask[u] |= 1u << (r & 31);
          steps += __popc(b);
        }
      }
    }
    if (__reduce_max_sync(DIAF_FULL, steps) * 10 < m * (k + 20)) {
      if (own)
        for (int p = 0; p < k; ++p) H[p + q * KP] = sc_zero<S>();
#pragma unroll
      for (int u = 0; u < NR; ++u) {
        uint32_t c = colmask[u];
        while (__any_sync(DIAF_FULL, c != 0)) {  // whole warp: the row masks come by shuffle
          const int r5 = c ? __ffs(c) - 1 : 0;
          uint32_t b = __shfl_sync(DIAF_FULL, rowmask[u], r5);
          if (c == 0) b = 0;
          const int r = DIAF_WARP * u + r5;
          const S x = b ? W[r + q * LDT] : sc_zero<S>();
          for (; b; b &= b - 1) {
            const int p = __ffs(b) - 1;
            H[p + q * KP] = sc_cmadd(H[p + q * KP], W[r + p * LDT], x);
          }
          c &= c - 1;
        }
      }
      __syncwarp();
      return;
    }
  }
  S acc[KMAX];
#pragma unroll
  for (int p = 0; p < KMAX; ++p) acc[p] = sc_zero<S>();
  if constexpr (kHalf) {
#pragma unroll
    for (int u = 0; u < NR; ++u) colmask[u] = 0;
  }
  if (own) {
    const S* wq = W + q * LDT;
    for (int r = kHalf ? lane >> 4 : 0; r < m; r += kHalf ? 2 : 1) {
      const S x = wq[r];
      if constexpr (kHalf)
        if (sc_real(x) != RealOf<S>(0) || sc_imag(x) != RealOf<S>(0)) colmask[r >> 5] |= 1u << (r & 31);
#pragma unroll
      for (int p = 0; p < KMAX; ++p)
        if (p < k) acc[p] = sc_cmadd(acc[p], W[r + p * LDT], x);
    }
  }
  if constexpr (kHalf) {
#pragma unroll
    for (int p = 0; p < KMAX; ++p) acc[p] += shfl_xor(acc[p], 16);
  }
  if (lane < k) {
#pragma unroll
    for (int p = 0; p < KMAX; ++p)
      if (p < k) H[p + lane * KP] = acc[p];
  }
  __syncwarp();
}

// Warp-wide sums of two values at once: the halves of the warp take one each
// after the first step (five FP64 additions instead of ten).
template <class T>
__device__ __forceinline__ void warp_sum2(T& a, T& b, int lane) {
  const bool up = lane >= 16;
  T v = up ? b : a;
  v += shfl_xor(up ? a : b, 16);
  v = group_sum<16>(v);
  a = shfl_idx(v, 0);
  b = shfl_idx(v, 16);
}

// Inverse of H - shift I for the Hermitian k x k matrix Hs (leading dimension
// KP; lane q reads column q) by symmetric sweeps without pivoting: the sweep
// on c replaces A_cc by -1/A_cc, A_ic by A_ic / A_cc and A_ij by
// A_ij - A_ic A_cj / A_cc, and after k of them A is minus the inverse; the
// pivots are the D of the LDL^* factorisation (their signs the inertia).
// A lane holds its column in registers, moved down by one row per sweep, so
// that the pivot row is always element 0 and one code body serves every
// sweep; a swept column is kept unscaled and its factor 1/pivot in *scale,
// so its update has the form of every other column's.  The pivot column is
// the conjugate of the pivot row, one entry per lane, and travels through buf
// (2 KMAX, 16-byte aligned, the halves alternating).  On return
// (H - shift I)^-1 has column `lane` -scale * a[KMAX - k ..).  *piv is the
// lane's pivot; returns the number of negative pivots.
template <class S, int KMAX, int KP>
__device__ __forceinline__ int warp_sweep_inverse(const S* Hs, RealOf<S> shift, int k, S (&a)[KMAX], S* buf, int lane,
                                                  RealOf<S>* piv, RealOf<S>* scale) {
  using R = RealOf<S>;
  constexpr int PV = 16 / (int)sizeof(S);
  static_assert(KMAX % PV == 0, "whole 16-byte packets");
#pragma unroll
  for (int i = 0; i < KMAX; ++i) {
    a[i] = (lane < k && i < k) ? Hs[i + lane * KP] : sc_zero<S>();
    if (i == lane && lane < k) a[i] -= sc_real_s<S>(shift);
  }
  int neg = 0;
  R sg = R(1);
#pragma unroll 1
  for (int c = 0; c < k; ++c) {
    const R p = __shfl_sync(DIAF_FULL, sc_real(a[0]), c);
    const R ri = R(1) / p;
    S* b = buf + (c & 1) * KMAX;
    int at = lane - c - 1;
    if (at < 0) at += KMAX;
    if (lane < KMAX) b[at] = sc_conj(sg * a[0]);
    __syncwarp();
    S u = ri * a[0];
    S tail = u;
    if (lane == c) {
      tail = sc_real_s<S>(R(-1));
      u = sc_zero<S>();
      sg = ri;
      *piv = p;
    }
    neg += p < R(0);
#pragma unroll
    for (int i0 = 0; i0 < KMAX; i0 += PV) {
      const Pack16<S> bb = *reinterpret_cast<const Pack16<S>*>(b + i0);
#pragma unroll
      for (int v = 0; v < PV; ++v)
        if (i0 + v + 1 < KMAX) a[i0 + v] = sc_msub(a[i0 + v + 1], bb.v[v], u);
    }
    a[KMAX - 1] = tail;
  }
  __syncwarp();
  *scale = sg;
  return neg;
}

// (H - shift I)^-1 x from warp_sweep_inverse's registers, one entry of x and
// of the result per lane; xb: KMAX scratch, 16-byte aligned.
template <class S, int KMAX>
__device__ __forceinline__ S warp_inverse_mul(const S (&a)[KMAX], RealOf<S> scale, S x, int k, S* xb, int lane) {
  constexpr int PV = 16 / (int)sizeof(S);
  int at = lane - k;
  if (at < 0) at += KMAX;
  if (lane < KMAX) xb[at] = lane < k ? x : sc_zero<S>();
  __syncwarp();
  S acc[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) acc[i] = sc_zero<S>();
#pragma unroll
  for (int i0 = 0; i0 < KMAX; i0 += PV) {
    const Pack16<S> bb = *reinterpret_cast<const Pack16<S>*>(xb + i0);
#pragma unroll
    for (int v = 0; v < PV; ++v) acc[(i0 + v) & 3] = sc_cmadd(acc[(i0 + v) & 3], a[i0 + v], bb.v[v]);
  }
  __syncwarp();
  return -scale * ((acc[0] + acc[1]) + (acc[2] + acc[3]));
}

// Ts: the tile (type SD, leading dimension LDT), Tw: a copy of it in the
// working type with the I_j rows zeroed (overwritten), rowmask: the columns
// that the lane's rows have (copy_tile), inI: the rows in I_j (>= 0), Hs: KP x
// KMAX scratch, gg / zz: KMAX / m scratch in SD.  The FP64 products run over the tile's nonzeros only
// (stencil tiles are 10 to 40 % full, and an FP64 instruction holds a sub-core
// for 64 cycles).  On success returns true and lane q < k has entry q of the
// unit vector in *x_out.
template <class S, class SD, int KMAX, int MMAX, int LDT, int KP>
__device__ bool warp_smallest_vector(const SD* Ts, const int32_t* inI, S* Tw,
                                     const uint32_t (&rowmask)[MMAX / DIAF_WARP], S* Hs, SD* gg, SD* zz, int m, int k,
                                     int lane, SD* x_out) {
  using R = RealOf<S>;
  static_assert(3 <= LDT, "the pivot columns and x fit the tile");
  if (k < 2 || m < k) return false;
  uint32_t colmask[MMAX / DIAF_WARP];
  tile_gram<S, KMAX, MMAX, LDT, KP>(Tw, rowmask, Hs, m, k, lane, colmask);
  S* buf = Tw;  // the tile has been read
  S* xs = buf + 2 * KMAX;
  R hrow = R(0), hqq = R(0);
  if (lane < k) {
    for (int p = 0; p < k; ++p) hrow += fabs(sc_real(Hs[p + lane * KP])) + fabs(sc_imag(Hs[p + lane * KP]));
    hqq = sc_real(Hs[lane + lane * KP]);
  }
  const R hinf = warp_max(hrow);
  // ---- inverse, conditioning, inverse iteration
  S inv[KMAX];
  R piv = R(1), scale = R(1);
  warp_sweep_inverse<S, KMAX, KP>(Hs, R(0), k, inv, buf, lane, &piv, &scale);
  constexpr R kmax = smallest_kappa_max<R>();
  if (!__all_sync(DIAF_FULL, lane >= k || (isfinite(hqq) && piv > R(0) && hqq <= kmax * kmax * piv))) return false;
  S x = lane < k ? sc_real_s<S>(R((lane * 37 + 11) % 17) - R(8.3)) : sc_zero<S>();
  R d = R(0);
#pragma unroll 1
  for (int it = 0; it < kInverseItMax; ++it) {
    const S y = warp_inverse_mul<S, KMAX>(inv, scale, x, k, xs, lane);
    const R nu = warp_sum(lane < k ? sc_real(sc_cmul(x, y)) : R(0));  // y^* H y
    const R ny = warp_sum(lane < k ? sc_abs2(y) : R(0));
    const R dn = nu / ny;
    x = rsqrt_r(ny) * y;
    const bool settled = it > 0 && fabs(dn - d) <= R(1e-2) * dn;
    d = dn;
    if (settled) break;
  }
  // ---- the shifted inverse and its inertia
  const R s = d + R(1.2e-5) * hinf;
  if (warp_sweep_inverse<S, KMAX, KP>(Hs, s, k, inv, buf, lane, &piv, &scale) != 1) return false;
  auto correction = [&](S r, R sh) -> S {  // -(H - d I)^-1 r, sh = s - d
    S dx = sc_zero<S>();
#pragma unroll 1
    for (int t = 0; t < 3; ++t) dx = warp_inverse_mul<S, KMAX>(inv, scale, -(r + sh * dx), k, xs, lane);
    return dx;
  };
  R last = R(1);
#pragma unroll 1
  for (int it = 0; it < 2; ++it) {
    if (lane < k) xs[lane] = x;
    __syncwarp();
    S hx = sc_zero<S>();
    if (lane < k)
      for (int p = 0; p < k; ++p) hx = sc_cmadd(hx, Hs[p + lane * KP], xs[p]);
    d = warp_sum(lane < k ? sc_real(sc_cmul(x, hx)) : R(0));
    S r = hx - d * x;
    if (lane >= k) r = sc_zero<S>();
    const S dx = correction(r, s - d);
    last = sqrt(warp_sum(lane < k ? sc_abs2(dx) : R(0)));
    x += dx;
    const R n2 = warp_sum(lane < k ? sc_abs2(x) : R(0));
    x = rsqrt_r(n2) * x;
    __syncwarp();
  }
  if (!(last <= R(0.05))) return false;
  // columns of A-hat that no chain of nonzeros of H ties to the vector's
  // largest entry are not part of it: exact zeros there, as the Jacobi (which
  // never rotates orthogonal columns) leaves them -- v_jj = 0 depends on it
  {
    uint32_t ties = 0;
    if (lane < k)
      for (int p = 0; p < k; ++p) ties |= sc_abs2(Hs[p + lane * KP]) != R(0) ? 1u << p : 0u;
    const R ax = lane < k ? sc_abs2(x) : R(-1);
    uint32_t comp = __ballot_sync(DIAF_FULL, ax == warp_max(ax));
    comp &= 0u - comp;
    for (uint32_t grown = 0; grown != comp;) {
      grown = comp;
      comp |= __reduce_or_sync(DIAF_FULL, (comp >> lane) & 1u ? ties : 0u);
    }
    if (!((comp >> lane) & 1u)) x = sc_zero<S>();
  }
  // ---- corrections against the FP64 tile
  using RD = RealOf<SD>;
  SD y = lane < k ? sc_cast<SD>(x) : sc_zero<SD>();
  R before = last;
  bool done = false;
#pragma unroll 1
  for (int it = 0; it < kCorrectMax && !done; ++it) {
    if (lane < k) gg[lane] = y;
    __syncwarp();
#pragma unroll
    for (int u = 0; u < MMAX / DIAF_WARP; ++u) {
      const int r = lane + DIAF_WARP * u;
      if (r < m) {
        SD z = sc_zero<SD>();
        for (uint32_t b = inI[r] < 0 ? rowmask[u] : 0u; b; b &= b - 1) {
          const int q = __ffs(b) - 1;
          z = sc_madd(z, Ts[r + q * LDT], gg[q]);
        }
        zz[r] = z;
      }
    }
    __syncwarp();
    SD g = sc_zero<SD>();
    {
      const int q = KMAX <= 16 ? lane & 15 : lane;
#pragma unroll
      for (int u = 0; u < MMAX / DIAF_WARP; ++u)
        for (uint32_t b = colmask[u]; b; b &= b - 1) {
          const int r = DIAF_WARP * u + __ffs(b) - 1;
          g = sc_cmadd(g, Ts[r + q * LDT], zz[r]);
        }
      if constexpr (KMAX <= 16) g += shfl_xor(g, 16);
    }
    RD yg = lane < k ? (RD)sc_real(sc_cmul(y, g)) : RD(0);
    RD yy = lane < k ? (RD)sc_abs2(y) : RD(0);
    warp_sum2(yg, yy, lane);
    RD iy = RD(2) - yy;  // 1 / yy, yy close to 1: Newton steps from 1
    iy *= fma(-yy, iy, RD(2));
    iy *= fma(-yy, iy, RD(2));
    const RD dd = yg * iy;
    const R room = R((RD)s - dd);  // at most the gap to the next eigenvalue
    if (!(room >= R(1.05e-5) * hinf && R(dd) > R(1e-24) * hinf)) return false;
    const S r = lane < k ? sc_cast<S>(g - dd * y) : sc_zero<S>();
    const S dx = correction(r, room);
    const R step = sqrt(warp_sum(lane < k ? sc_abs2(dx) : R(0)));
    if (lane < k) y += sc_cast<SD>(dx);
    // the next correction would be about step * (step / before)
    done = step * step <= R(kCorrectTol) * before;
    if (!done && it > 0 && !(step <= R(0.5) * before)) return false;
    before = step;
    __syncwarp();
  }
  if (!done) return false;
  const RD n2 = warp_sum(lane < k ? (RD)sc_abs2(y) : RD(0));
  RD inv2 = fma(RD(-0.5), n2, RD(1.5));  // 1 / sqrt(n2), n2 close to 1: Newton steps from 1
  inv2 *= fma(RD(-0.5) * n2 * inv2, inv2, RD(1.5));
  inv2 *= fma(RD(-0.5) * n2 * inv2, inv2, RD(1.5));
  *x_out = inv2 * y;
  return true;
}

// T w for the rows of the tile (w in wv) over its nonzeros: the rows in I_j to
// their places in vv, the sum of squares of the others (||A_j w - v||^2, as v
// takes the rows in I_j) returned.
template <class SD, int MMAX, int LDT>
__device__ __forceinline__ double split_rows(const SD* Ts, const int32_t* inI,
                                             const uint32_t (&rowmask)[MMAX / DIAF_WARP], const SD* wv, SD* vv, int m,
                                             int lane) {
  RealOf<SD> r2 = RealOf<SD>(0);
#pragma unroll
  for (int u = 0; u < MMAX / DIAF_WARP; ++u) {
    const int r = lane + DIAF_WARP * u;
    if (r >= m) continue;
    SD t = sc_zero<SD>();
    for (uint32_t b = rowmask[u]; b; b &= b - 1) {
      const int q = __ffs(b) - 1;
      t = sc_madd(t, Ts[r + q * LDT], wv[q]);
    }
    if (inI[r] >= 0) vv[inI[r]] = t;
    else r2 += sc_abs2(t);
  }
  return (double)warp_sum(r2);
}
