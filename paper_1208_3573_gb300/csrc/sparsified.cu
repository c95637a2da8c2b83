// Sparsified powers (Sec. 4.1, Algorithm 1): the W pattern from the
// truncated Neumann series of A^-1 D with the diagonal initial subspace,
// S = -D^-1 (A - D) (so that A = D (I - S)).  One warp per column j:
//
//   s = t = e_j;  for level = 1..k: t = S t, drop t by count p_l, s = s + t;
//   optionally drop s by count to `keep` entries (diagonal included).
//
// Dropping by count keeps the p largest-modulus off-diagonal entries (ties
// to the lower row); the diagonal entry j is never dropped and does not use
// up the count.  Exact-zero sums are not stored (the diagonal of s always is).
// Every sum is formed in a fixed order -- the products S_ic t_c of a row are
// added in increasing c, multiplications and additions rounded separately --
// so the values, and the choices made on them, do not depend on scheduling.
// The sparse vectors live in shared memory as row-sorted lists.  A first kernel
// takes the columns whose lists stay within 64 entries (the stencil operators:
// 36 products and 25 entries of a 7-point one): 3 KB per warp, products formed
// by all lanes, lists ordered by counting for every entry how many come before
// it (one pass of broadcast reads instead of a sorting network).  What does not
// fit goes to a second kernel with lists of up to kSpCap entries (22 KB per
// warp); a column that needs more reports DIAF_EUNSUPPORTED.  Both add in the
// same order.  Lognormal 64^3, keep 12: 5.9 ms a pass with the second kernel
// alone and two passes (count, fill); now 0.66 ms and one pass, which leaves the
// rows (the whole call 12.2 -> 0.78 ms).
#include <algorithm>
#include <atomic>
#include <cstdint>
#include <vector>

#include "factors.cuh"

namespace {

constexpr int kSpCap = 512;   // entries of a sparse vector / product list per warp
constexpr int kSpWarps = 2;   // warps per block

__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ Cx<double> mul_rn(Cx<double> a, Cx<double> b) {
  return {__dsub_rn(__dmul_rn(a.re, b.re), __dmul_rn(a.im, b.im)),
          __dadd_rn(__dmul_rn(a.re, b.im), __dmul_rn(a.im, b.re))};
}
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ Cx<double> add_rn(Cx<double> a, Cx<double> b) {
  return {__dadd_rn(a.re, b.re), __dadd_rn(a.im, b.im)};
}
__device__ __forceinline__ double neg(double a) { return -a; }
__device__ __forceinline__ Cx<double> neg(Cx<double> a) { return {-a.re, -a.im}; }
__device__ __forceinline__ bool is_zero_v(double a) { return a == 0.0; }
__device__ __forceinline__ bool is_zero_v(Cx<double> a) { return a.re == 0.0 && a.im == 0.0; }
// ordering key |v|^2, rounded step by step
__device__ __forceinline__ double key_of(double a) { return __dmul_rn(a, a); }
__device__ __forceinline__ double key_of(Cx<double> a) { return __dadd_rn(__dmul_rn(a.re, a.re), __dmul_rn(a.im, a.im)); }
__device__ __forceinline__ double recip(double d) { return 1.0 / d; }
__device__ __forceinline__ Cx<double> recip(Cx<double> d) {
  // 1/d = conj(d) / |d|^2 (only the exact structure matters for complex A)
  const double n2 = __dadd_rn(__dmul_rn(d.re, d.re), __dmul_rn(d.im, d.im));
  return {d.re / n2, -d.im / n2};
}

template <class S>
__global__ void diag_recip_kernel(int n, const int32_t* __restrict__ cp, const int32_t* __restrict__ ri,
                                  const S* __restrict__ v, S* __restrict__ dinv, uint32_t* status) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  S d = sc_zero<S>();
  bool found = false;
  for (int p = cp[i]; p < cp[i + 1]; ++p)
    if (ri[p] == i) { d = v[p]; found = true; }
  if (!found || is_zero_v(d)) atomicOr(status, DEV_ST_BAD_INPUT);
  dinv[i] = found ? recip(d) : sc_zero<S>();
}

template <class S>
struct SpWarp {
  int32_t tR[kSpCap];
  int32_t sR[kSpCap];
  uint64_t pK[kSpCap];
  int32_t keep[kSpCap];
  S tV[kSpCap];
  S sV[kSpCap];
  S pV[kSpCap];
};

// exclusive warp scan of x (lane order); returns the prefix, *total the sum
__device__ __forceinline__ int warp_excl_scan(int x, int lane, int* total) {
  int v = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(DIAF_FULL, v, o);
    if (lane >= o) v += y;
  }
  *total = __shfl_sync(DIAF_FULL, v, 31);
  return v - x;
}

// bitonic sort of pK[0..np) ascending with payload pV (np padded with ~0)
template <class S>
__device__ void warp_sort_pairs(SpWarp<S>& w, int np, int lane) {
  int P = 1;
  while (P < np) P <<= 1;
  for (int i = np + lane; i < P; i += 32) { w.pK[i] = ~0ull; w.pV[i] = sc_zero<S>(); }
  __syncwarp();
  for (int size = 2; size <= P; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int i = lane; i < P; i += 32) {
        const int jx = i ^ stride;
        if (jx > i) {
          const bool up = (i & size) == 0;
          const uint64_t a = w.pK[i], b = w.pK[jx];
          if ((a > b) == up) {
            w.pK[i] = b; w.pK[jx] = a;
            const S va = w.pV[i]; w.pV[i] = w.pV[jx]; w.pV[jx] = va;
          }
        }
      }
      __syncwarp();
    }
  }
}

// Sorted pairs (key = row << 32 | order) -> row-sorted list (R, V) of the
// sums over equal rows, added in key order; zero sums are dropped unless the
// row is `keep_row`.  Returns the list length.
template <class S>
__device__ int warp_segment_sums(const uint64_t* pK, const S* pV, int np, int32_t* R, S* V, int keep_row, int lane) {
  int carry = 0;
  for (int base = 0; base < np; base += 32) {
    const int p = base + lane;
    bool head = false, nz = false;
    int row = -1;
    S acc = sc_zero<S>();
    if (p < np) {
      row = (int)(pK[p] >> 32);
      head = p == 0 || (int)(pK[p - 1] >> 32) != row;
      if (head) {
        acc = pV[p];
        for (int q = p + 1; q < np && (int)(pK[q] >> 32) == row; ++q) acc = add_rn(acc, pV[q]);
        nz = !is_zero_v(acc) || row == keep_row;
      }
    }
    const unsigned bal = __ballot_sync(DIAF_FULL, head && nz);
    if (head && nz) {
      const int pos = carry + __popc(bal & ((1u << lane) - 1u));
      R[pos] = row;
      V[pos] = acc;
    }
    carry += __popc(bal);
  }
  __syncwarp();
  return carry;
}

// Keeps in (R, V, n) the entry `diag` (if present) and the `count` largest
// keys among the others (ties to the lower row); order preserved.  count < 0:
// keep all.  Returns the new length.
template <class S>
__device__ int warp_drop_by_count(SpWarp<S>& w, int32_t* R, S* V, int n, int diag, int count, int lane) {
  if (count < 0) return n;
  for (int i = lane; i < n; i += 32) w.keep[i] = R[i] == diag ? 1 : 0;
  __syncwarp();
  int off = 0;
  for (int i = lane; i < n; i += 32) off += R[i] != diag;
  off = warp_sum(off);
  if (off > count) {
    for (int it = 0; it < count; ++it) {  // select the best remaining entry, count times
      double bk = -1.0;
      int br = INT_MAX, bi = -1;
      for (int i = lane; i < n; i += 32) {
        if (w.keep[i] || R[i] == diag) continue;
        const double kk = key_of(V[i]);
        if (kk > bk || (kk == bk && R[i] < br)) { bk = kk; br = R[i]; bi = i; }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const double ok = __shfl_xor_sync(DIAF_FULL, bk, o);
        const int orr = __shfl_xor_sync(DIAF_FULL, br, o);
        const int oi = __shfl_xor_sync(DIAF_FULL, bi, o);
        if (ok > bk || (ok == bk && orr < br)) { bk = ok; br = orr; bi = oi; }
      }
      if (lane == 0 && bi >= 0) w.keep[bi] = 1;
      __syncwarp();
    }
  } else {
    for (int i = lane; i < n; i += 32) w.keep[i] = 1;
    __syncwarp();
  }
  // stable compaction
  int carry = 0;
  for (int base = 0; base < n; base += 32) {
    const int i = base + lane;
    const bool k = i < n && w.keep[i];
    int32_t r = 0;
    S v = sc_zero<S>();
    if (k) { r = R[i]; v = V[i]; }
    const unsigned bal = __ballot_sync(DIAF_FULL, k);
    __syncwarp();
    if (k) {
      const int pos = carry + __popc(bal & ((1u << lane) - 1u));
      R[pos] = r;
      V[pos] = v;
    }
    carry += __popc(bal);
    __syncwarp();
  }
  return carry;
}

// One column: returns its entry count (>= 0) and leaves the rows in w.sR, or
// -1 when a list would exceed kSpCap.
template <class S>
__device__ int sparsified_column(const int32_t* __restrict__ Acp, const int32_t* __restrict__ Ari,
                                 const S* __restrict__ Av, const S* __restrict__ dinv, int j, int k, int p_l,
                                 int keep, SpWarp<S>& w, int lane) {
  int nt = 1, ns = 1;
  if (lane == 0) {
    w.tR[0] = j; w.tV[0] = sc_real_s<S>(1.0);
    w.sR[0] = j; w.sV[0] = sc_real_s<S>(1.0);
  }
  __syncwarp();
  for (int level = 0; level < k; ++level) {
    // products S(:, c) t_c for the entries c of t, keyed (row, position of c in t)
    int np = 0, carry = 0;
    for (int base = 0; base < nt; base += 32) {
      const int e = base + lane;
      int cnt = 0;
      if (e < nt) {
        const int c = w.tR[e];
        cnt = Acp[c + 1] - Acp[c];
        for (int p = Acp[c]; p < Acp[c + 1]; ++p) cnt -= Ari[p] == c;
      }
      int tot;
      const int off = carry + warp_excl_scan(cnt, lane, &tot);
      if (carry + tot > kSpCap) return -1;  // warp-uniform
      if (e < nt) {
        const int c = w.tR[e];
        const S tc = w.tV[e];
        int o = off;
        for (int p = Acp[c]; p < Acp[c + 1]; ++p) {
          const int i = Ari[p];
          if (i == c) continue;
          const S sic = neg(mul_rn(dinv[i], Av[p]));  // S_ic = -(1/d_i) a_ic
          w.pK[o] = ((uint64_t)(uint32_t)i << 32) | (uint32_t)e;
          w.pV[o] = mul_rn(sic, tc);
          ++o;
        }
      }
      carry += tot;
    }
    np = carry;
    __syncwarp();
    warp_sort_pairs(w, np, lane);
    nt = warp_segment_sums(w.pK, w.pV, np, w.tR, w.tV, -1, lane);
    nt = warp_drop_by_count(w, w.tR, w.tV, nt, j, p_l > 0 ? p_l : -1, lane);
    // s = s + t: both row-sorted; s first so each sum is s_r + t_r
    if (ns + nt > kSpCap) return -1;
    for (int i = lane; i < ns; i += 32) { w.pK[i] = ((uint64_t)(uint32_t)w.sR[i] << 32); w.pV[i] = w.sV[i]; }
    for (int i = lane; i < nt; i += 32) { w.pK[ns + i] = ((uint64_t)(uint32_t)w.tR[i] << 32) | 1u; w.pV[ns + i] = w.tV[i]; }
    __syncwarp();
    warp_sort_pairs(w, ns + nt, lane);
    ns = warp_segment_sums(w.pK, w.pV, ns + nt, w.sR, w.sV, j, lane);
  }
  if (keep == 1) {  // the diagonal only
    int has = 0;
    for (int i = lane; i < ns; i += 32) has |= w.sR[i] == j;
    has = __any_sync(DIAF_FULL, has);
    __syncwarp();
    if (lane == 0 && has) w.sR[0] = j;
    __syncwarp();
    return has ? 1 : 0;
  }
  if (keep > 1) ns = warp_drop_by_count(w, w.sR, w.sV, ns, j, keep - 1, lane);
  return ns;
}

// ---- columns whose lists stay short
constexpr int kSmT = 32;     // entries of t
constexpr int kSmP = 64;     // products, or entries of s and t together
constexpr int kSmWarps = 8;  // warps per block
static_assert(kSmP == 64, "two entries per lane");

template <class S>
struct SpSmall {
  uint64_t uK[kSmP];  // as formed
  uint64_t pK[kSmP];  // ordered
  S uV[kSmP];
  S pV[kSmP];
  S tV[kSmT];
  S sV[kSmP];
  int32_t tR[kSmT];
  int32_t sR[kSmP];
  int32_t off[kSmT + 1];
};

// (uK, uV)[0 .. np) ordered by key into (pK, pV); keys are distinct but for
// the ~0 of unused places, which are left out.  Returns the entries placed.
template <class S>
__device__ int small_order(SpSmall<S>& w, int np, int lane) {
  const uint64_t k0 = lane < np ? w.uK[lane] : ~0ull, k1 = lane + 32 < np ? w.uK[lane + 32] : ~0ull;
  int r0 = 0, r1 = 0;
  for (int q = 0; q < np; ++q) {
    const uint64_t k = w.uK[q];
    r0 += k < k0;
    r1 += k < k1;
  }
  if (k0 != ~0ull) {
    w.pK[r0] = k0;
    w.pV[r0] = w.uV[lane];
  }
  if (k1 != ~0ull) {
    w.pK[r1] = k1;
    w.pV[r1] = w.uV[lane + 32];
  }
  const int placed = __popc(__ballot_sync(DIAF_FULL, k0 != ~0ull)) + __popc(__ballot_sync(DIAF_FULL, k1 != ~0ull));
  __syncwarp();
  return placed;
}

// warp_drop_by_count for a row-sorted list of at most kSmP entries, by ranks:
// keys are not negative, so they order like their bits (a NaN key is never
// among the best, as no comparison holds for it).
template <class S>
__device__ int small_drop_by_count(SpSmall<S>& w, int32_t* R, S* V, int n, int diag, int count, int lane) {
  if (count < 0) return n;
  int off = 0;
  uint64_t key[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int i = lane + 32 * u;
    key[u] = 0;
    if (i < n) {
      const double kk = key_of(V[i]);
      const bool other = R[i] != diag;
      off += other;
      key[u] = other && kk >= 0.0 ? (uint64_t)__double_as_longlong(kk) + 1 : 0;  // 0: not a candidate
      w.uK[i] = key[u];
    }
  }
  off = warp_sum(off);
  __syncwarp();
  bool kept[2];
  if (off > count) {
    int rank[2] = {0, 0};
    for (int q = 0; q < n; ++q) {
      const uint64_t k = w.uK[q];
#pragma unroll
      for (int u = 0; u < 2; ++u) rank[u] += k > key[u] || (k == key[u] && q < lane + 32 * u);
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int i = lane + 32 * u;
      kept[u] = i < n && (R[i] == diag || (key[u] != 0 && rank[u] < count));
    }
  } else {
    kept[0] = lane < n;
    kept[1] = lane + 32 < n;
  }
  int32_t r[2];
  S v[2];
#pragma unroll
  for (int u = 0; u < 2; ++u)
    if (kept[u]) {
      r[u] = R[lane + 32 * u];
      v[u] = V[lane + 32 * u];
    }
  __syncwarp();
  int carry = 0;
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const unsigned bal = __ballot_sync(DIAF_FULL, kept[u]);
    if (kept[u]) {
      const int pos = carry + __popc(bal & ((1u << lane) - 1u));
      R[pos] = r[u];
      V[pos] = v[u];
    }
    carry += __popc(bal);
  }
  __syncwarp();
  return carry;
}

// One column within the short lists: its entry count, the rows in w.sR, or -2
// when a list would be longer.
template <class S>
__device__ int small_column(const int32_t* __restrict__ Acp, const int32_t* __restrict__ Ari,
                            const S* __restrict__ Av, const S* __restrict__ dinv, int j, int k, int p_l, int keep,
                            SpSmall<S>& w, int lane) {
  int nt = 1, ns = 1;
  if (lane == 0) {
    w.tR[0] = j; w.tV[0] = sc_real_s<S>(1.0);
    w.sR[0] = j; w.sV[0] = sc_real_s<S>(1.0);
  }
  __syncwarp();
  for (int level = 0; level < k; ++level) {
    int c = 0, a0 = 0, len = 0;
    if (lane < nt) {
      c = w.tR[lane];
      a0 = Acp[c];
      len = Acp[c + 1] - a0;
    }
    int np;
    const int o = warp_excl_scan(len, lane, &np);
    if (np > kSmP) return -2;  // warp-uniform
    if (lane <= nt) w.off[lane] = o;  // lane nt: the total
    if (lane == 31 && nt == 32) w.off[32] = np;
    __syncwarp();
    for (int p = lane; p < np; p += 32) {  // product p: entry e of t, an entry of its column
      int e = 0;
      for (int hi = nt; hi - e > 1;) {
        const int mid = (e + hi) >> 1;
        if (w.off[mid] <= p) e = mid; else hi = mid;
      }
      const int cc = w.tR[e], q = Acp[cc] + p - w.off[e], i = Ari[q];
      if (i == cc) {
        w.uK[p] = ~0ull;
      } else {
        w.uK[p] = ((uint64_t)(uint32_t)i << 32) | (uint32_t)e;
        w.uV[p] = mul_rn(neg(mul_rn(dinv[i], Av[q])), w.tV[e]);  // S_ic t_c, S_ic = -(1/d_i) a_ic
      }
    }
    __syncwarp();
    const int nv = small_order(w, np, lane);
    // (a row list of at most nv entries: t's capacity is checked on the sums)
    int heads = 0;
    for (int p = lane; p < nv; p += 32) heads += p == 0 || (int)(w.pK[p - 1] >> 32) != (int)(w.pK[p] >> 32);
    if (warp_sum(heads) > kSmT) return -2;
    nt = warp_segment_sums(w.pK, w.pV, nv, w.tR, w.tV, -1, lane);
    nt = small_drop_by_count(w, w.tR, w.tV, nt, j, p_l > 0 ? p_l : -1, lane);
    if (ns + nt > kSmP) return -2;
    for (int i = lane; i < ns; i += 32) { w.uK[i] = ((uint64_t)(uint32_t)w.sR[i] << 32); w.uV[i] = w.sV[i]; }
    for (int i = lane; i < nt; i += 32) { w.uK[ns + i] = ((uint64_t)(uint32_t)w.tR[i] << 32) | 1u; w.uV[ns + i] = w.tV[i]; }
    __syncwarp();
    small_order(w, ns + nt, lane);
    ns = warp_segment_sums(w.pK, w.pV, ns + nt, w.sR, w.sV, j, lane);
  }
  if (keep > 0) ns = small_drop_by_count(w, w.sR, w.sV, ns, j, keep - 1, lane);
  return ns;
}

// What becomes of a finished column: its count, its rows at colptr[j], or its
// count and its rows at j * stride.
struct SpOut {
  const int32_t* colptr;
  int32_t* counts;
  int32_t* rowidx;
  int stride;
};
__device__ __forceinline__ void emit_column(const SpOut& out, int j, int cnt, const int32_t* rows, uint32_t* status,
                                            int lane) {
  if (cnt < 0) {
    if (lane == 0) {
      atomicOr(status, DEV_ST_CAPACITY);
      if (out.counts) out.counts[j] = 0;
    }
    return;
  }
  if (out.counts && lane == 0) out.counts[j] = cnt;
  if (!out.rowidx) return;
  size_t o = (size_t)j * out.stride;
  if (!out.counts) {
    o = out.colptr[j];
    if (out.colptr[j + 1] - (int)o != cnt) {  // the second pass must reproduce the first
      if (lane == 0) atomicOr(status, DEV_ST_BAD_INPUT);
      return;
    }
  }
  for (int i = lane; i < cnt; i += 32) out.rowidx[o + i] = rows[i];
}

template <class S>
__global__ void __launch_bounds__(kSmWarps * 32)
    sparsified_small_kernel(int n, const int32_t* __restrict__ Acp, const int32_t* __restrict__ Ari,
                            const S* __restrict__ Av, const S* __restrict__ dinv, int k, int p_l, int keep, SpOut out,
                            int32_t* list, int32_t* list_count, uint32_t* status) {
  extern __shared__ __align__(16) unsigned char sp_smem[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  SpSmall<S>& w = reinterpret_cast<SpSmall<S>*>(sp_smem)[wib];
  for (int j = blockIdx.x * kSmWarps + wib; j < n; j += gridDim.x * kSmWarps) {
    const int cnt = small_column<S>(Acp, Ari, Av, dinv, j, k, p_l, keep, w, lane);
    if (cnt == -2) {
      if (lane == 0) list[atomicAdd(list_count, 1)] = j;
    } else {
      emit_column(out, j, cnt, w.sR, status, lane);
    }
    __syncwarp();
  }
}

// The columns of the list (those the short lists could not hold).
template <class S>
__global__ void __launch_bounds__(kSpWarps * 32)
    sparsified_kernel(const int32_t* __restrict__ list, const int32_t* __restrict__ list_count,
                      const int32_t* __restrict__ Acp, const int32_t* __restrict__ Ari, const S* __restrict__ Av,
                      const S* __restrict__ dinv, int k, int p_l, int keep, SpOut out, uint32_t* status) {
  extern __shared__ __align__(16) unsigned char sp_smem[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  SpWarp<S>& w = reinterpret_cast<SpWarp<S>*>(sp_smem)[wib];
  const int count = *list_count;
  for (int idx = blockIdx.x * kSpWarps + wib; idx < count; idx += gridDim.x * kSpWarps) {
    const int j = list[idx];
    const int cnt = sparsified_column<S>(Acp, Ari, Av, dinv, j, k, p_l, keep, w, lane);
    emit_column(out, j, cnt, w.sR, status, lane);
    __syncwarp();
  }
}

__global__ void pack_columns_kernel(int n, int stride, const int32_t* __restrict__ rows,
                                    const int32_t* __restrict__ colptr, int32_t* __restrict__ rowidx) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int j = (int)(g / stride), i = (int)(g % stride);
  if (j >= n) return;
  const int o = colptr[j];
  if (i < colptr[j + 1] - o) rowidx[o + i] = rows[g];
}

template <class K>
cudaError_t allow_smem(K kern, size_t smem, std::atomic<uint64_t>& configured, int dev) {
  const uint64_t bit = 1ull << (dev & 63);  // the attribute is per device
  if (dev < 64 && (configured.load() & bit)) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) configured.fetch_or(bit);
  return e;
}

// Enqueues the pass over all columns; the caller reads *status (device) after it.
template <class S>
cudaError_t sparsified_enqueue(const diaf_csc* A, int k, int p_l, int keep, const SpOut& out, S* dinv, int32_t* list,
                               int32_t* list_count, uint32_t* status, cudaStream_t s) {
  const int n = A->n;
  const S* Av = (const S*)A->vals;
  cudaError_t e = cudaMemsetAsync(status, 0, sizeof(uint32_t), s);
  if (e == cudaSuccess) e = cudaMemsetAsync(list_count, 0, sizeof(int32_t), s);
  int dev = 0, sms = 152;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  diag_recip_kernel<S><<<ceil_div(n, 256), 256, 0, s>>>(n, A->colptr, A->rowidx, Av, dinv, status);
  DIAF_COUNT_LAUNCH();
  const size_t sm_small = sizeof(SpSmall<S>) * kSmWarps, sm_large = sizeof(SpWarp<S>) * kSpWarps;
  static std::atomic<uint64_t> conf_small{0}, conf_large{0};
  e = allow_smem(sparsified_small_kernel<S>, sm_small, conf_small, dev);
  if (e == cudaSuccess) e = allow_smem(sparsified_kernel<S>, sm_large, conf_large, dev);
  if (e != cudaSuccess) return e;
  const int blocks = std::min(ceil_div(n, kSmWarps), sms * 8);
  sparsified_small_kernel<S><<<blocks, kSmWarps * 32, sm_small, s>>>(n, A->colptr, A->rowidx, Av, dinv, k, p_l, keep,
                                                                     out, list, list_count, status);
  DIAF_COUNT_LAUNCH();
  const int blocks_l = std::min(ceil_div(n, kSpWarps), sms * 4);
  sparsified_kernel<S><<<blocks_l, kSpWarps * 32, sm_large, s>>>(list, list_count, A->colptr, A->rowidx, Av, dinv, k,
                                                                 p_l, keep, out, status);
  DIAF_COUNT_LAUNCH();
  return cudaGetLastError();
}

// Scratch of one call (stream-ordered, given back at its end).
struct Scratch {
  cudaStream_t s;
  std::vector<void*> held;
  explicit Scratch(cudaStream_t st) : s(st) {}
  template <class T>
  bool get(T** p, size_t count) {
    void* q = nullptr;
    if (cudaMallocAsync(&q, sizeof(T) * (count > 0 ? count : 1), s) != cudaSuccess) return false;
    held.push_back(q);
    *p = static_cast<T*>(q);
    return true;
  }
  ~Scratch() {
    for (void* p : held) cudaFreeAsync(p, s);
  }
};

// One pass; with d_colptr also the column pointers from the counts and nnz.
// Synchronises s.
diaf_status sparsified_pass(const diaf_csc* A, int k, int p_l, int keep, const int32_t* fill_colptr, int32_t* rowidx,
                            int stride, int32_t* d_colptr, int64_t* nnz, cudaStream_t s) {
  const int n = A->n;
  Scratch mem(s);
  uint32_t* status = nullptr;
  unsigned char* dinv = nullptr;
  int32_t *list = nullptr, *list_count = nullptr, *counts = nullptr, *bs = nullptr;
  const bool cplx = A->dtype == DIAF_C128;
  bool ok = mem.get(&status, 1) && mem.get(&dinv, (size_t)(cplx ? 16 : 8) * n) && mem.get(&list, n) &&
            mem.get(&list_count, 1);
  if (d_colptr) ok = ok && mem.get(&counts, n) && mem.get(&bs, scan_blocksums_size(n));
  if (!ok) return DIAF_ENOMEM;
  const SpOut out{fill_colptr, counts, rowidx, stride};
  cudaError_t e = cplx ? sparsified_enqueue<Cx<double>>(A, k, p_l, keep, out, (Cx<double>*)dinv, list, list_count,
                                                        status, s)
                       : sparsified_enqueue<double>(A, k, p_l, keep, out, (double*)dinv, list, list_count, status, s);
  uint32_t h = 0;
  int32_t last = 0;
  if (e == cudaSuccess && d_colptr) {
    e = exclusive_scan_i32(counts, d_colptr, n, bs, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&last, d_colptr + n, sizeof(int32_t), cudaMemcpyDeviceToHost, s);
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, status, sizeof(uint32_t), cudaMemcpyDeviceToHost, s);
  const cudaError_t se = cudaStreamSynchronize(s);
  if (e != cudaSuccess || se != cudaSuccess) return DIAF_ECUDA;
  if (h & DEV_ST_BAD_INPUT) {
    diaf_set_last_error("A has a zero or missing diagonal entry (or the passes disagree)");
    return DIAF_EINVAL;
  }
  if (h & DEV_ST_CAPACITY) {
    diaf_set_last_error("a column's product list exceeds 512 entries: use dropping by count (p_l)");
    return DIAF_EUNSUPPORTED;
  }
  if (nnz) *nnz = last;
  return DIAF_OK;
}

}  // namespace

extern "C" {

diaf_status diaf_sparsified_count(const diaf_csc* A, int32_t k, int32_t p_l, int32_t keep, int32_t* d_colptr,
                                  int64_t* nnz_out, void* stream) {
  if (!A || !d_colptr || !nnz_out || k < 0 || A->n < 0 || (A->dtype != DIAF_F64 && A->dtype != DIAF_C128))
    return DIAF_EINVAL;
  *nnz_out = 0;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (A->n == 0) return cudaMemsetAsync(d_colptr, 0, sizeof(int32_t), s) == cudaSuccess ? DIAF_OK : DIAF_ECUDA;
  return sparsified_pass(A, k, p_l, keep, nullptr, nullptr, 0, d_colptr, nnz_out, s);
}

diaf_status diaf_sparsified_fill(const diaf_csc* A, int32_t k, int32_t p_l, int32_t keep, const int32_t* d_colptr,
                                 int32_t* d_rowidx, void* stream) {
  if (!A || !d_colptr || k < 0 || A->n < 0 || (A->dtype != DIAF_F64 && A->dtype != DIAF_C128)) return DIAF_EINVAL;
  if (A->n == 0) return DIAF_OK;
  return sparsified_pass(A, k, p_l, keep, d_colptr, d_rowidx, 0, nullptr, nullptr, static_cast<cudaStream_t>(stream));
}

diaf_status diaf_sparsified_rows(const diaf_csc* A, int32_t k, int32_t p_l, int32_t keep, int32_t* d_rows,
                                 int32_t* d_colptr, int64_t* nnz_out, void* stream) {
  if (!A || !d_colptr || !nnz_out || k < 0 || keep < 1 || A->n < 0 || (A->n > 0 && !d_rows) ||
      (A->dtype != DIAF_F64 && A->dtype != DIAF_C128))
    return DIAF_EINVAL;
  *nnz_out = 0;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (A->n == 0) return cudaMemsetAsync(d_colptr, 0, sizeof(int32_t), s) == cudaSuccess ? DIAF_OK : DIAF_ECUDA;
  return sparsified_pass(A, k, p_l, keep, nullptr, d_rows, keep, d_colptr, nnz_out, s);
}

diaf_status diaf_sparsified_pack(int32_t n, int32_t keep, const int32_t* d_rows, const int32_t* d_colptr,
                                 int32_t* d_rowidx, void* stream) {
  if (n < 0 || keep < 1 || (n > 0 && (!d_rows || !d_colptr || !d_rowidx))) return DIAF_EINVAL;
  if (n == 0) return DIAF_OK;
  pack_columns_kernel<<<(unsigned)(((int64_t)n * keep + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      n, keep, d_rows, d_colptr, d_rowidx);
  DIAF_COUNT_LAUNCH();
  return cudaGetLastError() == cudaSuccess ? DIAF_OK : DIAF_ECUDA;
}

}  // extern "C"
