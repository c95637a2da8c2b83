// Four lanes per column: the mixed-precision DIAF-S (Sec. 2.2) for small real
// tiles (k_j <= 16, m_j <= 32, the size bucket of stencil operators).
//
// A quad of lanes runs the whole column -- gather, FP32 Householder QR of T,
// leverage keys, the V rule of Sec. 3.1, the smallest right singular vector of
// A-hat (T with the I_j rows removed), v = T(I_j,:) w, phase, FP64 residual
// and scatter -- with the same arithmetic as the warp kernel of
// column_mixed.cuh (the same FP32 factorisations, key-error bound, hand-back
// tests, and the method of smallest.cuh for the singular vector).  A warp
// works on eight columns at once: lane s of a quad owns the rows r = s (mod 4)
// of the tile and of every k x k matrix, so the per-column dependency chains
// carry two-step quad reductions instead of warp-wide ones, and no lane idles
// on the short vectors of these tiles.
//
// Storage: FP32 arrays in shared memory, element e of quad c at
// smem[32 (e / 4) + 8 (e mod 4) + c] (the 32 lanes of a warp reading four
// consecutive elements each hit 32 distinct banks); the FP64 tile in a global
// slab, four rows of one column side by side, interleaved across all quads of
// the grid (coalesced).  The kernel is instantiated for KMAX = 8, 13 and 16
// columns: the k x k matrices are swept and multiplied in registers with
// static indices (rows and columns from k on are an identity block), so a
// tile pays for KMAX columns.
//
// A column this kernel does not finish itself -- an empty or fixed-pattern
// column, a tile beyond its capacity or with fewer rows than columns, a tile
// too ill-conditioned for the FP32 factors, FP32 keys that cannot decide I_j,
// a smallest singular vector out of the direct method's reach -- goes to the
// defer list, which the warp kernel of column_mixed.cuh then runs (with its
// own FP64 keys, Jacobi and FP64 hand-back).
//
// What it replaced: a one-sided Jacobi SVD of the R of a second Householder QR
// took 52 % of the cycles and the correction in its basis 20 %.  Numeric pass on
// convection-diffusion 256^2 (25 x 13 tiles) 1.40 -> 0.72 ms, 843 -> 253 M
// instructions; power-law bucket 0 (k = 3 .. 16) 3.6 -> 2.2 ms.  What bounds it
// now is latency (30 % of the issue slots, 16 warps per SM by registers and by
// shared memory): waits on shared memory and shuffles, then on the slab, with
// 35 % of the cycles in the FP64 corrections (two passes over the tile at 1/64
// of the FP32 rate).
#pragma once

#include "column.cuh"

struct ThreadArgs {
  int M, K;              // capacity of this launch (rows, columns)
  double* slab;          // FP64 tile per quad of the grid: thread_slab_doubles each
  int nquads;            // quads of the grid (the slab's interleave)
  int32_t* defer_list;   // columns left to the warp kernel
  int32_t* defer_count;
};

constexpr int kThreadKMax = 16, kThreadMMax = 32;
constexpr int kQuad = 4;            // lanes per column
constexpr int kQuadCols = 8;        // columns per warp
constexpr int kQuadWarps = 1;       // warps per block

// Columns of the kernel instance for tiles of at most K columns.
__host__ __device__ constexpr int thread_instance(int K) { return K <= 8 ? 8 : (K <= 13 ? 13 : 16); }

// Shared-memory floats per column for capacity (M, K) of the KMAX instance:
// first the QR's M x K matrix, the keys (M) and the gather's K column ranges
// (8 bytes each, 8-byte aligned); then the rows of A-hat, 4 ceil(KMAX / 4)
// floats each; then H or its inverse (KMAX columns of 4 ceil(KMAX / 4) rows)
// and the FP64 vector x (KMAX), in whole groups of 4 elements.
__host__ __device__ constexpr int thread_arena_floats(int M, int K, int KMAX) {
  const int ku = (KMAX + 3) / 4;
  const int a = (M * K + M + 3) / 4 * 4 + 2 * ((K + 3) / 4 * 4);
  const int b = M * 4 * ku;
  const int c = 4 * ku * KMAX + 2 * 4 * ku;
  return a > b ? (a > c ? a : c) : (b > c ? b : c);
}
// FP64 slab doubles per quad: row r of column q at 4 ((r / 4) KMAX + q) + r mod 4.
__host__ __device__ constexpr int thread_slab_doubles(int M, int KMAX) { return (M + 3) / 4 * KMAX * 4; }
// Shared-memory bytes of one warp (eight columns).
__host__ __device__ constexpr size_t thread_warp_smem(int M, int K, int KMAX) {
  return sizeof(float) * (size_t)thread_arena_floats(M, K, KMAX) * 8;
}

// Element e of this quad's interleaved shared-memory array (base already
// offset by the quad's slot); element e + 4u lies at qptr(base, e)[32 u].
__device__ __forceinline__ float* qptr(float* base, int e) { return base + ((e >> 2) * 32 + (e & 3) * 8); }
__device__ __forceinline__ double* qptr(double* base, int e) { return base + ((e >> 2) * 32 + (e & 3) * 8); }
#define QS(base, e) (*qptr((base), (e)))

__device__ __forceinline__ float qsum(float v, unsigned qm) {
  v += __shfl_xor_sync(qm, v, 1);
  v += __shfl_xor_sync(qm, v, 2);
  return v;
}
__device__ __forceinline__ double qsum(double v, unsigned qm) {
  v += __shfl_xor_sync(qm, v, 1);
  v += __shfl_xor_sync(qm, v, 2);
  return v;
}

constexpr int kQR = kThreadMMax / 4;  // most rows a lane owns in a column of the tile
// Householder QR in place of the m x k column-major matrix at W (ld m,
// m >= k), FP32: reflector c maps W(c:m, c) to beta e_1 (the reflectors of
// warp_householder_qr).  Lane `sub` works on its rows (held in registers for
// the reflector's column); R ends in the upper triangle, visible to the whole
// quad on return.
__device__ __forceinline__ void quad_qr(float* W, int m, int k, int sub, unsigned qm) {
  for (int c = 0; c < k; ++c) {
    const int c0 = c * m;
    const int r0 = c + ((sub - c) & 3);  // first own row >= c
    float* pc = qptr(W, c0 + r0);
    float u[kQR];
    float s = 0.0f;
#pragma unroll
    for (int t = 0; t < kQR; ++t) {
      u[t] = r0 + 4 * t < m ? pc[32 * t] : 0.0f;
      s = fmaf(u[t], u[t], s);
    }
    s = qsum(s, qm);
    __syncwarp(qm);  // W(c, c), last written by its owner, is read by the whole quad
    const float alpha = QS(W, c0 + c);
    if (s == 0.0f) continue;
    const float ax = fabsf(alpha);
    const float nrm = sqrtf(s);
    const float ph = alpha < 0.0f ? -1.0f : 1.0f;
    const float two_uu = __fdividef(1.0f, nrm * (nrm + ax));
    if (r0 == c) u[0] = (ax + nrm) * ph;  // u_0 (the owner of row c)
    for (int q = c + 1; q < k; ++q) {
      float* pq = qptr(W, q * m + r0);
      float x[kQR];
      float f = 0.0f;
#pragma unroll
      for (int t = 0; t < kQR; ++t) {
        x[t] = r0 + 4 * t < m ? pq[32 * t] : 0.0f;
        f = fmaf(u[t], x[t], f);
      }
      f = qsum(f, qm) * two_uu;
#pragma unroll
      for (int t = 0; t < kQR; ++t)
        if (r0 + 4 * t < m) pq[32 * t] = fmaf(-f, u[t], x[t]);
    }
    if (r0 == c) pc[0] = -nrm * ph;  // beta
  }
  __syncwarp(qm);
}

// Inverse of H - shift I by symmetric sweeps (smallest.cuh), the rows spread
// over the quad: lane `sub` holds rows sub + 4u in a[u], moved one column to
// the left per sweep so that the pivot column is always element 0; a swept row
// is kept unscaled and its factor 1/pivot in sg[u].  The pivot row goes round
// by shuffles.  H: element (u, q) of lane `sub` at H[32 (u KMAX + q)] (base
// offset by 8 sub).  piv[u] receives the pivots; the inverse's row sub + 4u is
// -sg[u] a[u].
template <int KMAX>
__device__ __forceinline__ void quad_sweep_inverse(const float* H, float shift, float (&a)[(KMAX + 3) / 4][KMAX],
                                                   float (&piv)[(KMAX + 3) / 4], float (&sg)[(KMAX + 3) / 4], int sub,
                                                   unsigned qm) {
  constexpr int KU = (KMAX + 3) / 4;
#pragma unroll
  for (int u = 0; u < KU; ++u) {
    sg[u] = 1.0f;
    piv[u] = 1.0f;
#pragma unroll
    for (int q = 0; q < KMAX; ++q) {
      a[u][q] = H[32 * (u * KMAX + q)];
      if ((q >> 2) == u && (q & 3) == sub) a[u][q] -= shift;
    }
  }
#pragma unroll
  for (int uc = 0; uc < KU; ++uc) {  // pivot column c = 4 uc + sc
    constexpr int kLast = KMAX - 4 * (KU - 1);  // columns of the last group
#pragma unroll 1
    for (int sc = 0; sc < (uc == KU - 1 ? kLast : 4); ++sc) {
      float b[KMAX];
#pragma unroll
      for (int q = 0; q < KMAX; ++q) b[q] = __shfl_sync(qm, a[uc][q], sc, 4);
      const float ri = __fdividef(1.0f, b[0]);
      float f[KU];
#pragma unroll
      for (int u = 0; u < KU; ++u) f[u] = a[u][0] * ri;
      const bool own = sub == sc;
      const float tail = own ? -1.0f : f[uc];
      if (own) {
        piv[uc] = b[0];
        sg[uc] = ri;
        f[uc] = 0.0f;
      }
#pragma unroll
      for (int u = 0; u < KU; ++u) {
#pragma unroll
        for (int q = 0; q + 1 < KMAX; ++q) a[u][q] = fmaf(-f[u], b[q + 1], a[u][q + 1]);
        a[u][KMAX - 1] = u == uc ? tail : f[u];
      }
    }
  }
}

// y = (matrix) x for x and y spread over the quad like the rows; the lane's
// element (row sub + 4u, column q) in registers, or in shared memory at
// H[32 (u KMAX + q)].
template <int KMAX>
__device__ __forceinline__ void quad_mul_reg(const float (&a)[(KMAX + 3) / 4][KMAX], const float (&x)[(KMAX + 3) / 4],
                                             float (&y)[(KMAX + 3) / 4], unsigned qm) {
  constexpr int KU = (KMAX + 3) / 4;
  float t[KU];
#pragma unroll
  for (int u = 0; u < KU; ++u) t[u] = 0.0f;
#pragma unroll
  for (int q = 0; q < KMAX; ++q) {
    const float xq = __shfl_sync(qm, x[q >> 2], q & 3, 4);
#pragma unroll
    for (int u = 0; u < KU; ++u) t[u] = fmaf(a[u][q], xq, t[u]);
  }
#pragma unroll
  for (int u = 0; u < KU; ++u) y[u] = t[u];
}
template <int KMAX>
__device__ __forceinline__ void quad_mul_smem(const float* H, const float (&x)[(KMAX + 3) / 4],
                                              float (&y)[(KMAX + 3) / 4], unsigned qm) {
  constexpr int KU = (KMAX + 3) / 4;
  float t[KU];
#pragma unroll
  for (int u = 0; u < KU; ++u) t[u] = 0.0f;
#pragma unroll
  for (int q = 0; q < KMAX; ++q) {
    const float xq = __shfl_sync(qm, x[q >> 2], q & 3, 4);
#pragma unroll
    for (int u = 0; u < KU; ++u) t[u] = fmaf(H[32 * (u * KMAX + q)], xq, t[u]);
  }
#pragma unroll
  for (int u = 0; u < KU; ++u) y[u] = t[u];
}

template <int KU>
__device__ __forceinline__ float quad_dot(const float (&x)[KU], const float (&y)[KU], unsigned qm) {
  float s = 0.0f;
#pragma unroll
  for (int u = 0; u < KU; ++u) s = fmaf(x[u], y[u], s);
  return qsum(s, qm);
}

template <int KMAX>
__device__ void solve_column_quad(const ColArgs& a, const ThreadArgs& ta, int j, float* S, double* G, int sub,
                                  unsigned qm) {
  static_assert(KMAX <= kThreadKMax, "tile capacity");
  const int k = a.Wcp[j + 1] - a.Wcp[j];
  const int m = a.m[j];
  const int l = a.l[j];
  auto defer = [&]() {
    if (sub == 0) {
      const int pos = atomicAdd(ta.defer_count, 1);
      ta.defer_list[pos] = j;
    }
  };
  if (k == 0 || k > ta.K || k > KMAX || m > ta.M || m > kThreadMMax || m < k || l > m + 1 ||
      a.rule == DIAF_RULE_FIXED) {
    defer();
    return;
  }
  constexpr int KU = (KMAX + 3) / 4;  // rows of a k x k matrix a lane owns
  float* W = S;            // QR working matrix (ld m), keys from element HK on
  const int HK = ta.M * ta.K;
  // FP64 tile: rows 4t .. 4t + 3 of column q at G[(t KMAX + q) gstride .. + 3]
  const size_t gstride = (size_t)4 * ta.nquads;
  const int nown = (m - sub + 3) >> 2;  // own tile rows: sub, sub + 4, ...
  DIAF_PHASE_START();

  // ---- gather T = A(R_j, J_j): own rows zeroed, then each lane places every
  // fourth entry of the J_j columns by a binary search in R_j (a copy of R_j
  // in the keys' shared-memory slots, which are free until the keys)
  const int32_t* Rj = a.rows + a.Eoff[j];
  const int32_t* J = a.Wri + a.Wcp[j];
  const double* Av = reinterpret_cast<const double*>(a.Av);
  auto RS = [&](int r) -> int32_t& { return *reinterpret_cast<int32_t*>(qptr(W, HK + r)); };
  for (int r = sub; r < m; r += 4) RS(r) = Rj[r];
  // the entry range of A(:, J_j[q]) as an int pair behind the keys
  double* const C = reinterpret_cast<double*>(S - (threadIdx.x & 31) / 4) +
                    (size_t)((HK + ta.M + 3) / 4 * 4) * 4 + (threadIdx.x & 31) / 4;
  auto CR = [&](int q) -> int2& { return *reinterpret_cast<int2*>(qptr(C, q)); };
  for (int q = sub; q < k; q += 4) {
    const int c = J[q];
    CR(q) = make_int2(a.Acp[c], a.Acp[c + 1]);
  }
  for (int q = 0; q < k; ++q) {
    double* gq = G + q * gstride + sub;
    float* wq = qptr(W, q * m + sub);
#pragma unroll
    for (int t = 0; t < kQR; ++t)
      if (t < nown) {
        gq[t * KMAX * gstride] = 0.0;
        wq[32 * t] = 0.0f;
      }
  }
  __syncwarp(qm);
  uint32_t top = 0;
  for (int q = 0; q < k; ++q) {
    const int2 be = CR(q);
    for (int p = be.x + sub; p < be.y; p += 4) {
      const int32_t row = a.Ari[p];
      int r = 0;  // first position of R_j holding a row >= row (row is in R_j)
      for (int len = m; len > 0;) {
        const int half = len >> 1;
        if (RS(r + half) < row) {
          r += half + 1;
          len -= half + 1;
        } else {
          len = half;
        }
      }
      const double v = Av[p];
      top = max(top, top_word(v));
      G[((r >> 2) * KMAX + q) * gstride + (r & 3)] = v;
      QS(W, r + q * m) = (float)v;
    }
  }
  top = max(top, __shfl_xor_sync(qm, top, 1));
  top = max(top, __shfl_xor_sync(qm, top, 2));
  __syncwarp(qm);
  int unit;
  if (!tile_unit(top, &unit)) { defer(); return; }
  if (unit != 0) {
    for (int q = 0; q < k; ++q)
      for (int r = sub; r < m; r += 4) {
        double& g = G[((r >> 2) * KMAX + q) * gstride + (r & 3)];
        g *= pow2(-unit);
        QS(W, r + q * m) = (float)g;
      }
    __syncwarp(qm);
  }
  float cn[KMAX];
#pragma unroll
  for (int q = 0; q < KMAX; ++q) {
    float s2 = 0.0f;
    if (q < k) {
      const float* wq = qptr(W, q * m + sub);
#pragma unroll
      for (int t = 0; t < kQR; ++t)
        if (t < nown) s2 = fmaf(wq[32 * t], wq[32 * t], s2);
    }
    cn[q] = 0.0f;
    if (q < k) cn[q] = sqrtf(qsum(s2, qm));  // k is the same in the whole quad
  }

  // ---- FP32 QR of T and the conditioning estimate
  DIAF_PHASE(0);
  quad_qr(W, m, k, sub, qm);
  float kap = 0.0f;
  float rinv[KMAX];
#pragma unroll
  for (int q = 0; q < KMAX; ++q) {
    rinv[q] = 0.0f;
    if (q < k) {
      const float d = QS(W, q + q * m);
      kap = fmaxf(kap, scaled_kappa(cn[q], fabsf(d)));
      rinv[q] = __fdividef(1.0f, d);
    }
  }
  if (!(kap <= kMixedKappaMax)) { defer(); return; }

  // ---- leverage keys h_r = ||Q(r,:)||^2, Q = T R^-1 by rows (own rows; R's
  DIAF_PHASE(2);
  // column c read through four pointers, element c m + 4u + v at P[v][32 u])
  // two rows at a time: the loads of R are shared and the two solves are
  // independent chains
  for (int t = 0; t < nown; t += 2) {
    const int r = sub + 4 * t;
    const bool two = t + 1 < nown;
    float z[KMAX], y[KMAX];
    float h = 0.0f, h1 = 0.0f;
    const double* g0 = G + t * KMAX * gstride + sub;
    const double* g1 = g0 + KMAX * gstride;
#pragma unroll
    for (int c = 0; c < KMAX; ++c, g0 += gstride, g1 += gstride) {
      z[c] = 0.0f;
      y[c] = 0.0f;
      if (c < k) {
        const float* P0 = qptr(W, c * m);
        const float* P1 = qptr(W, c * m + 1);
        const float* P2 = qptr(W, c * m + 2);
        const float* P3 = qptr(W, c * m + 3);
        float acc = (float)*g0;
        float acc1 = two ? (float)*g1 : 0.0f;
#pragma unroll
        for (int p2 = 0; p2 < c; ++p2) {
          const float* P = (p2 & 3) == 0 ? P0 : ((p2 & 3) == 1 ? P1 : ((p2 & 3) == 2 ? P2 : P3));
          const float rv = P[32 * (p2 >> 2)];
          acc = fmaf(-z[p2], rv, acc);
          acc1 = fmaf(-y[p2], rv, acc1);
        }
        z[c] = acc * rinv[c];
        y[c] = acc1 * rinv[c];
        h = fmaf(z[c], z[c], h);
        h1 = fmaf(y[c], y[c], h1);
      }
    }
    QS(W, HK + r) = h;
    if (two) QS(W, HK + r + 4) = h1;
  }
  __syncwarp(qm);

  // ---- I_j: the diagonal plus the l - 1 admissible rows of largest key
  DIAF_PHASE(3);
  // (ties within tau to the lower row), as select_rows_greedy; every lane of
  // the quad takes the same decisions (picks as bits)
  uint32_t adm = 0;
  for (int r = 0; r < m; ++r)
    if (admissible_row(a.rule, Rj[r], j, a.blk)) adm |= 1u << r;
  uint32_t picked = 0;
  float margin = FLT_MAX;
  const float tau = (float)a.tie_tol;
  for (int t = 0; t < l - 1; ++t) {
    const uint32_t cand = adm & ~picked;
    float hm = -FLT_MAX;
    for (uint32_t b = cand; b; b &= b - 1) hm = fmaxf(hm, QS(W, HK + __ffs(b) - 1));
    int rmax = INT_MAX;
    for (uint32_t b = cand; b && rmax == INT_MAX; b &= b - 1)
      if (QS(W, HK + __ffs(b) - 1) == hm) rmax = __ffs(b) - 1;
    const float thr = hm - tau;
    int best = INT_MAX;
    for (uint32_t b = cand; b; b &= b - 1) {
      const int r = __ffs(b) - 1;
      const float h = QS(W, HK + r);
      if (r != rmax) margin = fminf(margin, fabsf(h - thr));
      if (h >= thr && best == INT_MAX) best = r;
    }
    if (best == INT_MAX && cand) best = __ffs(cand) - 1;  // no key reaches the threshold (non-finite keys)
    if (best < m) picked |= 1u << best;
  }
  if (l > 1) {
    const double delta = kMixedDeltaScale * (m + k) * (double)FLT_EPSILON * (double)kap;
    if ((double)margin <= 2.0 * delta) { defer(); return; }  // FP32 keys cannot decide this column
  }
  // I_j = the picked tile rows, row j, and j itself when it is not a tile row
  // (inserted in order); tile row r in I_j has position pos_of(r)
  uint32_t inI = picked;
  int rj = -1;
  for (int r = 0; r < m; ++r)
    if (Rj[r] == j) rj = r;
  if (rj >= 0) inI |= 1u << rj;
  const bool jin = a.jin[j] != 0;
  int jbefore = m;  // tile rows from this index on come after an inserted j
  if (!jin) {
    jbefore = 0;
    while (jbefore < m && Rj[jbefore] < j) ++jbefore;
  }
  auto below = [](int r) { return r >= 32 ? 0xffffffffu : (1u << r) - 1u; };  // bits of the rows below r
  auto pos_of = [&](int r) { return __popc(inI & below(r)) + ((!jin && r >= jbefore) ? 1 : 0); };
  if (__popc(inI) + (jin ? 0 : 1) != l || (jin && rj < 0)) { defer(); return; }  // not reached
  const int v0 = a.Vcp[j];
  const int jpos = jin ? pos_of(rj) : __popc(inI & below(jbefore));
  if (sub == 0 && !jin) a.Vri[v0 + jpos] = j;
  for (int r = sub; r < m; r += 4)
    if ((inI >> r) & 1u) a.Vri[v0 + pos_of(r)] = Rj[r];

  // ---- A-hat's rows in FP32 (the I_j rows zeroed), row-major in groups of 4
  DIAF_PHASE(4);
  __syncwarp(qm);  // the keys and the QR's matrix have been read
  for (int t = 0; t < nown; ++t) {
    const int r = sub + 4 * t;
    const bool out = (inI >> r) & 1u;
    const double* g = G + t * KMAX * gstride + sub;
    float* row = S + r * KU * 32;
#pragma unroll
    for (int q = 0; q < 4 * KU; ++q, g += gstride) {
      float v = 0.0f;
      if (q < KMAX && q < k && !out) v = (float)*g;
      row[(q >> 2) * 32 + (q & 3) * 8] = v;
    }
  }
  __syncwarp(qm);
  // ---- H = A-hat^T A-hat: the lane's rows sub + 4u
  DIAF_PHASE(6);
  float a4[KU][KMAX];
#pragma unroll
  for (int u = 0; u < KU; ++u)
#pragma unroll
    for (int q = 0; q < KMAX; ++q) a4[u][q] = 0.0f;
  for (int r = 0; r < m; ++r) {
    const float* row = S + r * KU * 32;
    float own[KU];
#pragma unroll
    for (int u = 0; u < KU; ++u) own[u] = row[u * 32 + sub * 8];
#pragma unroll
    for (int q = 0; q < KMAX; ++q) {
      const float v = row[(q >> 2) * 32 + (q & 3) * 8];
#pragma unroll
      for (int u = 0; u < KU; ++u) a4[u][q] = fmaf(own[u], v, a4[u][q]);
    }
  }
  __syncwarp(qm);  // the rows have been read
  float hinf = 0.0f, hd[KU];
#pragma unroll
  for (int u = 0; u < KU; ++u) {
    float hs = 0.0f;
    hd[u] = 0.0f;
#pragma unroll
    for (int q = 0; q < KMAX; ++q) {
      hs += fabsf(a4[u][q]);
      if ((q >> 2) == u && (q & 3) == sub) hd[u] = a4[u][q];
    }
    hinf = fmaxf(hinf, hs);
  }
  hinf = fmaxf(hinf, __shfl_xor_sync(qm, hinf, 1));
  hinf = fmaxf(hinf, __shfl_xor_sync(qm, hinf, 2));
  // an exactly zero column of A-hat (all its entries in I_j) is an exact zero
  // singular value with w = e_c: only the gap to the others is left to check
  uint32_t zeros = 0;
  float* const Hs = S + sub * 8;
#pragma unroll
  for (int u = 0; u < KU; ++u) {
    const int row = sub + 4 * u;
    const bool zero = row < k && hd[u] == 0.0f;
    if (zero) zeros |= 1u << row;
    const bool pad = zero || row >= k;  // those rows: a diagonal of the others' size
    if (pad) hd[u] = hinf;
#pragma unroll
    for (int q = 0; q < KMAX; ++q)
      Hs[32 * (u * KMAX + q)] = (pad && (q >> 2) == u && (q & 3) == sub) ? hinf : a4[u][q];
  }
  zeros |= __shfl_xor_sync(qm, zeros, 1);
  zeros |= __shfl_xor_sync(qm, zeros, 2);
  if ((zeros & (zeros - 1u)) != 0 || !(hinf > 0.0f)) { defer(); return; }
  float piv[KU], sg[KU], x[KU];
  float s = 1.2e-5f * hinf;  // the shift; d is added unless there is a zero column
  auto conditioned = [&]() {  // column-scaled kappa <= kGramKappaMax from the pivots
    bool ok = true;
#pragma unroll
    for (int u = 0; u < KU; ++u)
      ok &= sub + 4 * u >= k || (piv[u] > 0.0f && hd[u] <= kGramKappaMax * kGramKappaMax * piv[u]);
    return (__ballot_sync(qm, ok) & qm) == qm;
  };
  if (zeros == 0) {
    DIAF_PHASE(5);
    quad_sweep_inverse<KMAX>(Hs, 0.0f, a4, piv, sg, sub, qm);
    if (!conditioned()) { defer(); return; }
#pragma unroll
    for (int u = 0; u < KU; ++u) x[u] = sub + 4 * u < k ? (float)(((sub + 4 * u) * 37 + 11) % 17) - 8.3f : 0.0f;
    float d = 0.0f;
#pragma unroll 1
    for (int it = 0; it < kInverseItMax; ++it) {
      float y[KU];
      quad_mul_reg<KMAX>(a4, x, y, qm);
#pragma unroll
      for (int u = 0; u < KU; ++u) y[u] *= -sg[u];
      const float nu = quad_dot<KU>(x, y, qm), ny = quad_dot<KU>(y, y, qm);
      const float dn = __fdividef(nu, ny), inv = rsqrtf(ny);
#pragma unroll
      for (int u = 0; u < KU; ++u) x[u] = inv * y[u];
      const bool settled = it > 0 && fabsf(dn - d) <= 1e-2f * dn;
      d = dn;
      if (settled) break;
    }
    s += d;
  }
  // ---- the shifted inverse and its inertia: exactly one eigenvalue below s
  // (none but the zero column's, which the diagonal above stands in for)
  quad_sweep_inverse<KMAX>(Hs, s, a4, piv, sg, sub, qm);
  if (zeros != 0) {
    if (!conditioned()) { defer(); return; }
  } else {
    int neg = 0;
#pragma unroll
    for (int u = 0; u < KU; ++u) neg += piv[u] < 0.0f;
    neg += __shfl_xor_sync(qm, neg, 1);
    neg += __shfl_xor_sync(qm, neg, 2);
    if (neg != 1) { defer(); return; }
  }
  DIAF_PHASE(7);
  double xd[KU];  // the vector in FP64, entries sub + 4u
  double* const X = reinterpret_cast<double*>(S - (threadIdx.x & 31) / 4) + 16 * KU * KMAX + (threadIdx.x & 31) / 4;
  uint32_t flags = 0;
  if (zeros != 0) {
#pragma unroll
    for (int u = 0; u < KU; ++u) xd[u] = (zeros >> (sub + 4 * u)) & 1u ? 1.0 : 0.0;
  } else {
    // the inverse itself in a4 (its rows' factors applied)
#pragma unroll
    for (int u = 0; u < KU; ++u)
#pragma unroll
      for (int q = 0; q < KMAX; ++q) a4[u][q] *= -sg[u];
    float last = 1.0f;
#pragma unroll 1
    for (int it = 0; it < 2; ++it) {
      float hx[KU], dx[KU];
      quad_mul_smem<KMAX>(Hs, x, hx, qm);
      const float d = quad_dot<KU>(x, hx, qm);
#pragma unroll
      for (int u = 0; u < KU; ++u) hx[u] -= d * x[u];
      // -(H - d I)^-1 r by two Neumann steps on the shifted inverse
      const float sh = s - d;
#pragma unroll
      for (int u = 0; u < KU; ++u) dx[u] = 0.0f;
#pragma unroll 1
      for (int n = 0; n < 3; ++n) {
#pragma unroll
        for (int u = 0; u < KU; ++u) dx[u] = -fmaf(sh, dx[u], hx[u]);
        quad_mul_reg<KMAX>(a4, dx, dx, qm);
      }
      last = sqrtf(quad_dot<KU>(dx, dx, qm));
#pragma unroll
      for (int u = 0; u < KU; ++u) x[u] += dx[u];
      const float inv = rsqrtf(quad_dot<KU>(x, x, qm));
#pragma unroll
      for (int u = 0; u < KU; ++u) x[u] *= inv;
    }
    if (!(last <= 0.05f)) { defer(); return; }
    // columns that no chain of nonzeros of H ties to the largest entry: exact zeros
    {
      uint32_t ties[KU];
      float ax = -1.0f;
#pragma unroll
      for (int u = 0; u < KU; ++u) {
        ties[u] = 0;
#pragma unroll
        for (int q = 0; q < KMAX; ++q)
          if (q < k && Hs[32 * (u * KMAX + q)] != 0.0f) ties[u] |= 1u << q;
        if (sub + 4 * u >= k) ties[u] = 0;
        else ax = fmaxf(ax, fabsf(x[u]));
      }
      float am = fmaxf(ax, __shfl_xor_sync(qm, ax, 1));
      am = fmaxf(am, __shfl_xor_sync(qm, am, 2));
      uint32_t comp = 0;
#pragma unroll
      for (int u = 0; u < KU; ++u)
        if (sub + 4 * u < k && fabsf(x[u]) == am) comp |= 1u << (sub + 4 * u);
      comp |= __shfl_xor_sync(qm, comp, 1);
      comp |= __shfl_xor_sync(qm, comp, 2);
      comp &= 0u - comp;
      for (uint32_t grown = 0; grown != comp;) {
        grown = comp;
#pragma unroll
        for (int u = 0; u < KU; ++u)
          if ((grown >> (sub + 4 * u)) & 1u) comp |= ties[u];
        comp |= __shfl_xor_sync(qm, comp, 1);
        comp |= __shfl_xor_sync(qm, comp, 2);
      }
#pragma unroll
      for (int u = 0; u < KU; ++u) xd[u] = (comp >> (sub + 4 * u)) & 1u ? (double)x[u] : 0.0;
    }
    __syncwarp(qm);  // H has been read: the inverse takes its place
#pragma unroll
    for (int u = 0; u < KU; ++u)
#pragma unroll
      for (int q = 0; q < KMAX; ++q) Hs[32 * (u * KMAX + q)] = a4[u][q];
    // ---- corrections against the FP64 tile: one pass over it gives both
    // z = A-hat x on the lane's rows and its part of g = A-hat^T z, which the
    // quad's lanes then sum and split
    double before = (double)last;
    bool done = false;
#pragma unroll 1
    for (int it = 0; it < kCorrectMax && !done; ++it) {
#pragma unroll
      for (int u = 0; u < KU; ++u) X[32 * u + 8 * sub] = xd[u];
      __syncwarp(qm);
      double g[4 * KU], zz = 0.0;
#pragma unroll
      for (int q = 0; q < 4 * KU; ++q) g[q] = 0.0;
      for (int t = 0; t < nown; ++t) {
        if ((inI >> (sub + 4 * t)) & 1u) continue;
        const double* gp = G + t * KMAX * gstride + sub;
        double tv[KMAX], z = 0.0;
#pragma unroll
        for (int q = 0; q < KMAX; ++q, gp += gstride) {
          tv[q] = q < k ? *gp : 0.0;
          z = fma(tv[q], X[(q >> 2) * 32 + (q & 3) * 8], z);
        }
        zz = fma(z, z, zz);
#pragma unroll
        for (int q = 0; q < KMAX; ++q) g[q] = fma(tv[q], z, g[q]);
      }
      __syncwarp(qm);
      // own entries of g: halves exchanged with lane ^ 1, then with lane ^ 2
      double go[KU];
#pragma unroll
      for (int u = 0; u < KU; ++u) {
        double h[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const double g0 = g[4 * u + 2 * e], g1 = g[4 * u + 2 * e + 1];
          h[e] = ((sub & 1) ? g1 : g0) + __shfl_xor_sync(qm, (sub & 1) ? g0 : g1, 1);
        }
        go[u] = ((sub & 2) ? h[1] : h[0]) + __shfl_xor_sync(qm, (sub & 2) ? h[0] : h[1], 2);
      }
      double xx = 0.0;
#pragma unroll
      for (int u = 0; u < KU; ++u) xx = fma(xd[u], xd[u], xx);
      xx = qsum(xx, qm);
      double ix = 2.0 - xx;  // 1 / xx, xx close to 1: two Newton steps from 1
      ix *= fma(-xx, ix, 2.0);
      ix *= fma(-xx, ix, 2.0);
      const double d = qsum(zz, qm) * ix;
      const double room = (double)s - d;  // at most the gap to the next eigenvalue
      if (!(room >= 1.05e-5 * (double)hinf && d > 1e-24 * (double)hinf)) { defer(); return; }
      float r[KU], dx[KU];
#pragma unroll
      for (int u = 0; u < KU; ++u) r[u] = (float)fma(-d, xd[u], go[u]);
#pragma unroll
      for (int u = 0; u < KU; ++u) dx[u] = 0.0f;
#pragma unroll 1
      for (int n = 0; n < 3; ++n) {
#pragma unroll
        for (int u = 0; u < KU; ++u) dx[u] = -fmaf((float)room, dx[u], r[u]);
        quad_mul_smem<KMAX>(Hs, dx, dx, qm);
      }
      const double step = sqrtf(quad_dot<KU>(dx, dx, qm));
#pragma unroll
      for (int u = 0; u < KU; ++u) xd[u] += (double)dx[u];
      done = step * step <= kCorrectTol * before;  // the next correction: about step (step / before)
      if (!done && it > 0 && !(step <= 0.5 * before)) { defer(); return; }
      before = step;
    }
    if (!done) { defer(); return; }
    double xn2 = 0.0;
#pragma unroll
    for (int u = 0; u < KU; ++u) xn2 = fma(xd[u], xd[u], xn2);
    xn2 = qsum(xn2, qm);
    double inv = 1.5 - 0.5 * xn2;  // 1 / sqrt(xn2), xn2 within 1e-2 of 1: Newton steps from 1
    inv *= fma(-0.5 * xn2 * inv, inv, 1.5);
    inv *= fma(-0.5 * xn2 * inv, inv, 1.5);
#pragma unroll
    for (int u = 0; u < KU; ++u) xd[u] *= inv;
  }
#pragma unroll
  for (int u = 0; u < KU; ++u) X[32 * u + 8 * sub] = xd[u];
  __syncwarp(qm);

  // ---- v = T(I_j,:) w (into V's values by the row owners), phase v_jj >= 0,
  DIAF_PHASE(8);
  // FP64 residual
  double* Vout = reinterpret_cast<double*>(a.Vv) + v0;
  double vn2 = 0.0, vjj = 0.0, r2 = 0.0;
  if (sub == 0 && !jin) Vout[jpos] = 0.0;
  // rows in I_j: v_r = (T w)_r, so their term of ||T w - v|| is exactly zero;
  // the other rows contribute (T w)_r (the residual from its definition)
  for (int t = 0; t < nown; ++t) {
    const int r = sub + 4 * t;
    double sv = 0.0;
    const double* gp = G + t * KMAX * gstride + sub;
    for (int q = 0; q < k; ++q, gp += gstride) sv = fma(*gp, QS(X, q), sv);
    if ((inI >> r) & 1u) {
      Vout[pos_of(r)] = sv;
      vn2 = fma(sv, sv, vn2);
      if (r == rj) vjj = sv;
    } else {
      r2 = fma(sv, sv, r2);
    }
  }
  vn2 = qsum(vn2, qm);
  vjj = qsum(vjj, qm);
  double ph = 1.0;
  const double zl = 64.0 * DBL_EPSILON;
  if (vjj * vjj > zl * zl * vn2) {
    ph = vjj < 0.0 ? -1.0 : 1.0;
  } else {
    flags |= DIAF_FLAG_VJJ_ZERO;
    double amx = 0.0, wsel = 1.0;
    for (int q = 0; q < k; ++q) {
      const double xq = QS(X, q);
      if (fabs(xq) > amx) { amx = fabs(xq); wsel = xq; }
    }
    ph = wsel < 0.0 ? -1.0 : 1.0;
  }
  bool finite = true;
  const double pv = copysign(pow2(unit), ph);
  for (int t = 0; t < nown; ++t) {
    const int r = sub + 4 * t;
    if ((inI >> r) & 1u) {
      const int pos = pos_of(r);
      const double vt = pv * Vout[pos];
      Vout[pos] = vt;
      finite &= isfinite(vt);
    }
  }
  r2 = qsum(r2, qm);
  const double resj = sqrt(r2);
  // (no zero column: sigma_min > 1e-12 sigma_max; ||H||_inf <= k sigma_max^2)
  if (zeros != 0 && resj <= 1e-14 * (double)sqrtf(hinf / (float)k)) flags |= DIAF_FLAG_RANK_DEFICIENT;
  finite &= isfinite(resj);
  double* Wout = reinterpret_cast<double*>(a.Wv) + a.Wcp[j];
  for (int q = sub; q < k; q += 4) {
    const double wq = ph * QS(X, q);
    finite &= isfinite(wq);
    Wout[q] = wq;
  }
  const unsigned fin = __ballot_sync(qm, finite) & qm;
  if (fin != qm) flags |= DIAF_FLAG_NONFINITE;
  if (sub == 0) {
    a.res[j] = unit != 0 ? pow2(unit) * resj : resj;
    a.flags[j] = flags | a.extra_flags;
  }
  if (a.Hri) {  // the final I_j to the host (the rows as written above), then the column's word
    if (sub == 0 && !jin) a.Hri[v0 + jpos] = j;
    for (int r = sub; r < m; r += 4)
      if ((inI >> r) & 1u) a.Hri[v0 + pos_of(r)] = Rj[r];
    __threadfence_system();
    __syncwarp(qm);
    if (sub == 0) store_release_sys(a.Hgen + j, a.gen);
  }
  DIAF_PHASE(9);
}

// The persistent loop: each warp takes eight columns of the list at a time,
// one per quad.
template <int KMAX>
__global__ void __launch_bounds__(32 * kQuadWarps, 16) column_thread_kernel(ColArgs a, ThreadArgs ta) {
  extern __shared__ __align__(16) float tsmem[];
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int sub = lane & 3, slot = lane >> 2;
  const unsigned qm = 0xFu << (lane & ~3);
  const int gq = (blockIdx.x * kQuadWarps + warp) * kQuadCols + slot;  // quad index in the grid
  float* S = tsmem + (size_t)warp * thread_arena_floats(ta.M, ta.K, KMAX) * 8 + slot;
  double* G = ta.slab + (size_t)4 * gq;
  const int count = *a.list_count;
  while (true) {
    int base = 0;
    if (lane == 0) base = atomicAdd(a.work_counter, kQuadCols);
    base = __shfl_sync(DIAF_FULL, base, 0);
    if (base >= count) break;
    const int idx = base + slot;
    if (idx < count) solve_column_quad<KMAX>(a, ta, list_at(a, count, idx), S, G, sub, qm);
    __syncwarp();
  }
}

#undef QS
