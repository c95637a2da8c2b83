// Row-oriented sparse operations for the solve phase.
#include <atomic>
#include <climits>
#include <type_traits>

#include "plan.cuh"
#include "sparse.cuh"

namespace {

// CSC -> CSR.  kConvLanes lanes per column count the entries of every row
// and, after the scan, place them (independent loads and atomics across the
// lanes: the columns are short, so one thread per column would serialise
// them); the atomics leave each row's entries in no particular order, so one
// warp per row then sorts them by column.
constexpr int kConvLanes = 8;

__global__ void count_rows_kernel(int n, const int32_t* __restrict__ cp, const int32_t* __restrict__ ri,
                                  int32_t* __restrict__ cnt) {
  const int64_t gid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int j = (int)(gid / kConvLanes), sub = (int)(gid % kConvLanes);
  if (j >= n) return;
  const int e = cp[j + 1];
  for (int p = cp[j] + sub; p < e; p += kConvLanes) atomicAdd(&cnt[ri[p]], 1);
}

template <class S>
__global__ void fill_rows_kernel(int n, const int32_t* __restrict__ cp, const int32_t* __restrict__ ri,
                                 const S* __restrict__ v, const int32_t* __restrict__ rowptr,
                                 int32_t* __restrict__ cursor, int32_t* __restrict__ colidx, S* __restrict__ vals) {
  const int64_t gid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int j = (int)(gid / kConvLanes), sub = (int)(gid % kConvLanes);
  if (j >= n) return;
  const int e = cp[j + 1];
  for (int p = cp[j] + sub; p < e; p += kConvLanes) {
    const int i = ri[p];
    const int pos = rowptr[i] + atomicAdd(&cursor[i], 1);
    colidx[pos] = j;
    vals[pos] = v[p];
  }
}

// One warp per row: a row of up to 32 entries is sorted by column with a
// bitonic network of shuffles (each value follows its column through its
// source position); a longer row by insertion sort in lane 0.  The result is
// the same whatever order the atomics left.
template <class S>
__global__ void sort_rows_kernel(int n, const int32_t* __restrict__ rowptr, int32_t* __restrict__ colidx,
                                 S* __restrict__ vals) {
  const int row = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (row >= n) return;  // whole warps: blockDim.x is a multiple of 32
  const int a = rowptr[row], len = rowptr[row + 1] - a;
  if (len <= 1) return;
  if (len <= 32) {
    int key = lane < len ? colidx[a + lane] : INT_MAX;
    int src = lane;
    for (int size = 2; size <= 32; size <<= 1) {
      for (int stride = size >> 1; stride > 0; stride >>= 1) {
        const int ok = __shfl_xor_sync(DIAF_FULL, key, stride);
        const int os = __shfl_xor_sync(DIAF_FULL, src, stride);
        const bool keep_min = ((lane & stride) == 0) == ((lane & size) == 0);
        const bool less = ok < key || (ok == key && os < src);  // (ok, os) before (key, src)
        if (keep_min ? less : !less) {
          key = ok;
          src = os;
        }
      }
    }
    S v = sc_zero<S>();
    if (lane < len) v = vals[a + src];
    __syncwarp();
    if (lane < len) {
      colidx[a + lane] = key;
      vals[a + lane] = v;
    }
  } else if (lane == 0) {
    for (int p = a + 1; p < a + len; ++p) {
      const int c = colidx[p];
      const S v = vals[p];
      int q = p - 1;
      while (q >= a && colidx[q] > c) {
        colidx[q + 1] = colidx[q];
        vals[q + 1] = vals[q];
        --q;
      }
      colidx[q + 1] = c;
      vals[q + 1] = v;
    }
  }
}

template <class S>
cudaError_t csc_to_csr_t(int n, int64_t nnz, const int32_t* cp, const int32_t* ri, const S* v, int32_t* rowptr,
                         int32_t* colidx, S* vals, int32_t* work, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  int32_t* cnt = work;
  int32_t* bs = work + n;
  const int lane_blocks = (int)(((int64_t)n * kConvLanes + 255) / 256);
  cudaMemsetAsync(cnt, 0, sizeof(int32_t) * n, s);
  count_rows_kernel<<<lane_blocks, 256, 0, s>>>(n, cp, ri, cnt);
  DIAF_COUNT_LAUNCH();
  exclusive_scan_i32(cnt, rowptr, n, bs, s);
  cudaMemsetAsync(cnt, 0, sizeof(int32_t) * n, s);
  fill_rows_kernel<S><<<lane_blocks, 256, 0, s>>>(n, cp, ri, v, rowptr, cnt, colidx, vals);
  DIAF_COUNT_LAUNCH();
  sort_rows_kernel<S><<<ceil_div(n, 8), 256, 0, s>>>(n, rowptr, colidx, vals);
  DIAF_COUNT_LAUNCH();
  return cudaGetLastError();
}

// y = M x with a group of G lanes per row.
template <class S, int G>
__global__ void spmv_kernel(int n, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colidx,
                            const S* __restrict__ vals, const S* __restrict__ x, S* __restrict__ y) {
  int gid = (blockIdx.x * blockDim.x + threadIdx.x);
  int row = gid / G, sub = gid % G;
  S acc = sc_zero<S>();
  if (row < n) {
    for (int p = rowptr[row] + sub; p < rowptr[row + 1]; p += G) acc += vals[p] * x[colidx[p]];
  }
  acc = group_sum<G>(acc);
  if (row < n && sub == 0) y[row] = acc;
}

constexpr int kLevelThreads = 1024;
constexpr int kLevelPtrSmem = 8192;  // level pointers kept in shared memory up to this many levels
constexpr int kPrefetch = 4;         // off-diagonal entries of a row held in registers ahead of its level

template <class S>
constexpr int level_window() { return 131072 / (int)sizeof(S); }  // 128 KB ring

// Row i of V goes to level position p = lvlptr[lev i] + rank i (the walk's
// place of row i in its level); len[p] = its number of off-diagonal entries.
__global__ void level_place_kernel(int n, const int32_t* __restrict__ lev, const int32_t* __restrict__ rank,
                                   const int32_t* __restrict__ rcnt, const int32_t* __restrict__ lvlptr,
                                   int32_t* __restrict__ pos, int32_t* __restrict__ xrow, int32_t* __restrict__ len,
                                   int32_t* __restrict__ poff, double* __restrict__ pval) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int p = lvlptr[lev[i]] + rank[i];
  pos[i] = p;
  xrow[p] = i;
  if (poff) {  // every place empty; its value is read all the same (times zero)
    reinterpret_cast<int4*>(poff)[p] = make_int4(-1, -1, -1, -1);
    double2* const v = reinterpret_cast<double2*>(pval) + 2 * (size_t)p;
    v[0] = v[1] = make_double2(0.0, 0.0);
  } else {
    len[p] = rcnt[i];
  }
}

// V's rows level by level, straight from its columns: kConvLanes lanes per
// column j; entry (i, j), i != j, goes to slot slot[e] of row position
// pos[i] with column position pos[j] and value v_ij / v_ii (the row scaled by
// its diagonal, which sits at entry dpos[i] of column i); the diagonal entry
// gives 1/v_jj at position pos[j] and raises *zflag when it is zero (or not
// a number).
template <class S>
__global__ void level_fill_kernel(int n, const int32_t* __restrict__ cp, const int32_t* __restrict__ ri,
                                  const S* __restrict__ v, const int32_t* __restrict__ dpos,
                                  const int32_t* __restrict__ slot, const int32_t* __restrict__ pos,
                                  const int32_t* __restrict__ rowptr, int32_t* __restrict__ pcol,
                                  S* __restrict__ pval, S* __restrict__ pdinv, uint32_t* __restrict__ zflag) {
  const int64_t gid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int j = (int)(gid / kConvLanes), sub = (int)(gid % kConvLanes);
  if (j >= n) return;
  const int e1 = cp[j + 1];
  for (int e = cp[j] + sub; e < e1; e += kConvLanes) {
    const int i = ri[e];
    if (i == j) {
      const S d = v[e];
      if (!(sc_abs2(d) > 0.0)) atomicOr(zflag, 1u);
      pdinv[pos[j]] = (1.0 / sc_abs2(d)) * sc_conj(d);
    } else {
      const S d = v[dpos[i]];
      const int q = rowptr[pos[i]] + slot[e];
      pcol[q] = pos[j];
      pval[q] = ((1.0 / sc_abs2(d)) * sc_conj(d)) * v[e];
    }
  }
}

// The same for a real V in the packed form: entry slot[e] of the row.
__global__ void packed_fill_kernel(int n, const int32_t* __restrict__ cp, const int32_t* __restrict__ ri,
                                   const double* __restrict__ v, const int32_t* __restrict__ dpos,
                                   const int32_t* __restrict__ slot, const int32_t* __restrict__ pos,
                                   const int32_t* __restrict__ lev, const int32_t* __restrict__ lvlptr, int r, int nlev,
                                   int32_t* __restrict__ poff, double* __restrict__ pval, double* __restrict__ pdinv,
                                   uint32_t* __restrict__ zflag, uint32_t* __restrict__ pflags) {
  const int64_t gid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int j = (int)(gid / kConvLanes), sub = (int)(gid % kConvLanes);
  if (j >= n) return;
  const int e1 = cp[j + 1];
  for (int e = cp[j] + sub; e < e1; e += kConvLanes) {
    const int i = ri[e];
    const double d = i == j ? v[e] : v[dpos[i]];
    if (i == j) {
      if (!(d * d > 0.0)) atomicOr(zflag, 1u);
      pdinv[pos[j]] = (1.0 / (d * d)) * d;
    } else {
      const int pi = pos[i], pj = pos[j];
      const size_t q = (size_t)kPackEntries * pi + slot[e];
      poff[q] = pj;
      pval[q] = ((1.0 / (d * d)) * d) * v[e];
      const int last = (lev[i] / r + 1) * r;  // the end of the row's group
      if (pj < lvlptr[last < nlev ? last : nlev] - level_window<double>()) atomicOr(pflags, kPackFar);
    }
  }
}

// A complex V's packed form (r = 1) from its level-ordered rows: copied, so
// that the solve's results keep every bit (the residual at which a restarted
// GMRES stops moves by 1e-6 of itself with the last bit of the apply).
__global__ void pack_rows_kernel(int nlev, const int32_t* __restrict__ lvlptr, const int32_t* __restrict__ rowptr,
                                 const int32_t* __restrict__ colidx, const Cx<double>* __restrict__ vals,
                                 int32_t* __restrict__ poff, Cx<double>* __restrict__ pval, uint32_t* pflags) {
  for (int l = blockIdx.x; l < nlev; l += gridDim.x) {
    const int e = lvlptr[l + 1];
    for (int p = lvlptr[l] + (int)threadIdx.x; p < e; p += blockDim.x) {
      const int a = rowptr[p], len = rowptr[p + 1] - a;
      for (int q = 0; q < kPackEntries; ++q) {
        const int c = q < len ? colidx[a + q] : -1;
        poff[(size_t)kPackEntries * p + q] = c;
        pval[(size_t)kPackEntries * p + q] = q < len ? vals[a + q] : sc_zero<Cx<double>>();
        if (c >= 0 && c < e - level_window<Cx<double>>()) atomicOr(pflags, kPackFar);
      }
    }
  }
}

// t[p] = x[xrow[p]] / diag of row p (level order): the scaled right-hand
// side the level solves start from, for all rows at once.
template <class S>
__global__ void scale_rhs_kernel(int n, const S* __restrict__ dinv, const int32_t* __restrict__ xrow,
                                 const S* __restrict__ x, S* __restrict__ t) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < n) t[p] = dinv[p] * x[xrow[p]];
}

__global__ void remap_cols_kernel(int64_t nnz, const int32_t* __restrict__ pos, const int32_t* __restrict__ cin,
                                  int32_t* __restrict__ cout) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz; e += (int64_t)gridDim.x * blockDim.x)
    cout[e] = pos[cin[e]];
}

// Level-scheduled solve on the level-ordered matrix: the rows of level l are
// the contiguous positions lvlptr[l]..lvlptr[l+1], their off-diagonal
// entries point at positions of earlier levels, t is kept in level order.
// The rows are stored scaled by 1/diag and t starts as the scaled right-hand
// side (scale_rhs_kernel), so a row is t[p] -= sum v_pj t[j] in place, with
// no multiplication after the sum.  Nothing a row needs except t of earlier
// levels depends on the solve, so every thread loads its next row (bounds,
// its start value t[p] and the first kPrefetch entries) before the barrier
// that ends the current level; after the barrier only the loads of t remain
// on the critical path.  Those come from a ring of the last kWin
// positions of t in shared memory: while level [b, e) is written, slots of
// positions >= e - kWin are not overwritten, so reads of such positions use
// the ring and older ones use t in global memory (written too).
// One pass of the block over everything the solve will read (level-ordered
// rows and the start values in t), with 16-byte loads (the library's own
// arrays are 256-byte aligned).  The first solve after the level-ordered
// copies were built ran 0.42 ms instead of 0.29 ms on the 256^2
// convection-diffusion V, and a second solve right after it at full speed:
// the data was cold for the one SM that runs the solve.  With this pass
// (~30 us) in front, the first solve takes 0.35 ms; later solves skip it.
template <class S>
__device__ __forceinline__ void warm_level_data(int n, int nnz, const int32_t* rowptr, const int32_t* colidx,
                                                const S* vals, S* t) {
  unsigned acc = 0;
  const int4* r4 = reinterpret_cast<const int4*>(rowptr);
  const int4* c4 = reinterpret_cast<const int4*>(colidx);
  const int4* v4 = reinterpret_cast<const int4*>(vals);
  const int4* t4 = reinterpret_cast<const int4*>(t);
  for (int i = threadIdx.x; i < n / 4; i += blockDim.x) acc += r4[i].x;
  for (int i = threadIdx.x; i < nnz / 4; i += blockDim.x) acc += c4[i].z;
  for (int i = threadIdx.x; i < (int)(n * sizeof(S) / 16); i += blockDim.x) acc += t4[i].w;
  for (int i = threadIdx.x; i < (int)(nnz * sizeof(S) / 16); i += blockDim.x) acc += v4[i].y;
  if (acc == 0x9e3779b9u && n < 0) t[0] = sc_zero<S>();  // keeps the loads; never taken
}

template <class S>
__global__ void __launch_bounds__(kLevelThreads, 1)
    trsv_levels_perm_kernel(int nlev, const int32_t* __restrict__ lvlptr, const int32_t* __restrict__ rowptr,
                            const int32_t* __restrict__ colidx, const S* __restrict__ vals,
                            S* t, int warm) {
  constexpr int kWin = level_window<S>();
  static_assert((kWin & (kWin - 1)) == 0, "ring size must be a power of two");
  extern __shared__ __align__(16) unsigned char level_ring[];
  S* tw = reinterpret_cast<S*>(level_ring);
  __shared__ int32_t sptr[kLevelPtrSmem + 1];
  const bool in_smem = nlev <= kLevelPtrSmem;
  if (in_smem)
    for (int i = threadIdx.x; i <= nlev; i += blockDim.x) sptr[i] = lvlptr[i];
  if (warm) {
    const int n_ = lvlptr[nlev];
    warm_level_data<S>(n_, rowptr[n_], rowptr, colidx, vals, t);
  }
  __syncthreads();
#define DIAF_LP(l) (in_smem ? sptr[(l)] : lvlptr[(l)])
  // registers for the first row this thread takes in the coming level
  int rb = 0, re = 0;
  S xb = sc_zero<S>();
  int pc[kPrefetch];
  S pv[kPrefetch];
#define DIAF_FETCH(pp)                                 \
  do {                                                 \
    const int p_ = (pp);                               \
    rb = rowptr[p_];                                   \
    re = rowptr[p_ + 1];                               \
    xb = t[p_];                                        \
    _Pragma("unroll") for (int q = 0; q < kPrefetch; ++q) { \
      const bool in = rb + q < re;                     \
      pc[q] = in ? colidx[rb + q] : 0;                 \
      pv[q] = in ? vals[rb + q] : sc_zero<S>();        \
    }                                                  \
  } while (0)
  if (nlev > 0 && DIAF_LP(0) + (int)threadIdx.x < DIAF_LP(1)) DIAF_FETCH(DIAF_LP(0) + (int)threadIdx.x);
  for (int lv = 0; lv < nlev; ++lv) {
    const int b = DIAF_LP(lv), e = DIAF_LP(lv + 1);
    const int lo = e - kWin;  // ring holds positions >= lo unchanged during this level
#define DIAF_TGET(c) ((c) >= lo ? tw[(c) & (kWin - 1)] : t[(c)])
    int p = b + threadIdx.x;
    if (p < e) {
      S acc = xb;
#pragma unroll
      for (int q = 0; q < kPrefetch; ++q)
        if (rb + q < re) acc = sc_msub(acc, pv[q], DIAF_TGET(pc[q]));
      for (int k = rb + kPrefetch; k < re; ++k) acc = sc_msub(acc, vals[k], DIAF_TGET(colidx[k]));
      t[p] = acc;
      tw[p & (kWin - 1)] = acc;
    }
    for (p += blockDim.x; p < e; p += blockDim.x) {  // levels wider than the block
      S acc = t[p];
      for (int k = rowptr[p]; k < rowptr[p + 1]; ++k) acc = sc_msub(acc, vals[k], DIAF_TGET(colidx[k]));
      t[p] = acc;
      tw[p & (kWin - 1)] = acc;
    }
    if (lv + 1 < nlev) {
      const int nb = e, ne = DIAF_LP(lv + 2);
      if (nb + (int)threadIdx.x < ne) DIAF_FETCH(nb + (int)threadIdx.x);
    }
    __syncthreads();
#undef DIAF_TGET
  }
#undef DIAF_FETCH
#undef DIAF_LP
}

// The same solve for matrices whose levels are at most kDeepThreads rows
// wide, with the row data fetched kDeep levels ahead instead of one.  A
// thread keeps its rows of the next kDeep levels in kDeep register sets (set
// k: the levels lv with lv mod kDeep = k).  A row's loads form two dependent
// round trips (the bounds in rowptr; then the entries and the start value
// t[p]), issued one level apart -- the first right after the set's previous level is done, the
// second one level later -- so no thread waits on a load before a barrier.
constexpr int kDeepThreads = 256;
constexpr int kDeep = 4;

template <class S>
__global__ void __launch_bounds__(kDeepThreads, 1)
    trsv_levels_deep_kernel(int nlev, const int32_t* __restrict__ lvlptr, const int32_t* __restrict__ rowptr,
                            const int32_t* __restrict__ colidx, const S* __restrict__ vals,
                            S* t, int warm) {
  constexpr int kWin = level_window<S>();
  extern __shared__ __align__(16) unsigned char level_ring[];
  S* tw = reinterpret_cast<S*>(level_ring);
  __shared__ int32_t sptr[kLevelPtrSmem + 1];
  const bool in_smem = nlev <= kLevelPtrSmem;
  if (in_smem)
    for (int i = threadIdx.x; i <= nlev; i += blockDim.x) sptr[i] = lvlptr[i];
  if (warm) {
    const int n_ = lvlptr[nlev];
    warm_level_data<S>(n_, rowptr[n_], rowptr, colidx, vals, t);
  }
  __syncthreads();
#define DIAF_LP(l) (in_smem ? sptr[(l)] : lvlptr[(l)])
  int rb[kDeep], re[kDeep], xr[kDeep];
  S xb[kDeep];
  int pc[kDeep][kPrefetch];
  S pv[kDeep][kPrefetch];
  // first round trip: the row's bounds (xr = its position, -1: no row)
#define DIAF_STAGE_A(k, lvl)                                      \
  do {                                                            \
    rb[k] = 0;                                                    \
    re[k] = 0;                                                    \
    xr[k] = -1;                                                   \
    const int p_ = DIAF_LP(lvl) + (int)threadIdx.x;               \
    if (p_ < DIAF_LP((lvl) + 1)) {                                \
      rb[k] = rowptr[p_];                                         \
      re[k] = rowptr[p_ + 1];                                     \
      xr[k] = p_;                                                 \
    }                                                             \
  } while (0)
  // second round trip: the start value t[p] and the first kPrefetch entries
#define DIAF_STAGE_B(k)                                           \
  do {                                                            \
    if (xr[k] >= 0) {                                             \
      xb[k] = t[xr[k]];                                           \
      _Pragma("unroll") for (int q = 0; q < kPrefetch; ++q) {     \
        const bool in = rb[k] + q < re[k];                        \
        pc[k][q] = in ? colidx[rb[k] + q] : 0;                    \
        pv[k][q] = in ? vals[rb[k] + q] : sc_zero<S>();           \
      }                                                           \
    }                                                             \
  } while (0)
#pragma unroll
  for (int k = 0; k < kDeep; ++k)
    if (k < nlev) DIAF_STAGE_A(k, k);
#pragma unroll
  for (int k = 0; k < kDeep; ++k)
    if (k < nlev) DIAF_STAGE_B(k);
  for (int lv0 = 0; lv0 < nlev; lv0 += kDeep) {
#pragma unroll
    for (int k = 0; k < kDeep; ++k) {
      const int lv = lv0 + k;
      if (lv < nlev) {  // uniform over the block
        const int b = DIAF_LP(lv), e = DIAF_LP(lv + 1);
        const int lo = e - kWin;
#define DIAF_TGET(c) ((c) >= lo ? tw[(c) & (kWin - 1)] : t[(c)])
        const int p = b + (int)threadIdx.x;
        if (p < e) {
          S acc = xb[k];
#pragma unroll
          for (int q = 0; q < kPrefetch; ++q)
            if (rb[k] + q < re[k]) acc = sc_msub(acc, pv[k][q], DIAF_TGET(pc[k][q]));
          for (int j = rb[k] + kPrefetch; j < re[k]; ++j) acc = sc_msub(acc, vals[j], DIAF_TGET(colidx[j]));
          t[p] = acc;
          tw[p & (kWin - 1)] = acc;
        }
#undef DIAF_TGET
        if (lv + kDeep < nlev) DIAF_STAGE_A(k, lv + kDeep);
        // the set whose first round trip was issued one level ago
        const int kb = (k + kDeep - 1) % kDeep;
        if (lv >= 1 && lv + kDeep - 1 < nlev) DIAF_STAGE_B(kb);
        __syncthreads();
      }
    }
  }
#undef DIAF_STAGE_A
#undef DIAF_STAGE_B
#undef DIAF_LP
}

// ---- the packed form: levels in groups
//
// On the single solving SM a level cost about 0.58 us whatever its width: the
// chain barrier - bounds - column indices - t - FP64 - barrier, some 150
// instructions long, not the arithmetic (convection-diffusion 256^2: 512
// levels of 128 rows, 0.30 ms, where the FP64 pipe needs 0.03).  Two changes:
//
// a row's entries at fixed places (two to five 16-byte loads, issued groups
// ahead), so that between two barriers a thread only reads t from the ring,
// multiplies and writes its own t;
//
// r = 4 levels between two barriers.  Eliminating the rows of its own group
// from a row, t_i = x'_i + sum C_ik t_k has only k of earlier groups.  The
// coefficients C are formed once (merge_kernel); x' is the right-hand side put
// through the group's own block, group by group independently of each other,
// so all SMs do it at once (group_rhs_kernel).  The stencil operators' rows
// have 2 entries and 3.3 merged ones (at most 5), so the chip's one FP64 pipe
// that solves does 1.7 times the work for a quarter of the barriers.  Complex
// rows (4 entries, 8 merged) are bound by that pipe: they keep r = 1.

// The merged entries of group blockIdx.x, level by level: the row's own
// entries of earlier groups, and for each entry of its own group v times that
// row's merged entries.  Products beyond kMergeMax (or not numbers) are not
// formed into a solve: infinite, they would turn the zeros of a sparse
// right-hand side into NaN, which the level by level solve does not.
constexpr uint32_t kMergeMax = 0x54b249adu;  // top_word(1e100)
__global__ void __launch_bounds__(256) merge_kernel(int nlev, int r, const int32_t* __restrict__ lvlptr,
                                                    const int32_t* __restrict__ poff, const double* __restrict__ pval,
                                                    int32_t* mpos, int32_t* moff, double* mval, uint32_t* pflags) {
  const int l0 = blockIdx.x * r;
  const int l1 = l0 + r < nlev ? l0 + r : nlev;
  const int gs = lvlptr[l0];
  for (int l = l0; l < l1; ++l) {
    const int e = lvlptr[l + 1];
    for (int p = lvlptr[l] + (int)threadIdx.x; p < e; p += blockDim.x) {
      int32_t c[kMergeEntries];
      double v[kMergeEntries];
#pragma unroll
      for (int q = 0; q < kMergeEntries; ++q) {
        c[q] = -1;
        v[q] = 0.0;
      }
      bool full = false;
      auto add = [&](int32_t col, double val) {
        bool placed = false;
#pragma unroll
        for (int q = 0; q < kMergeEntries; ++q)
          if (!placed && (c[q] < 0 || c[q] == col)) {
            c[q] = col;
            v[q] += val;
            placed = true;
          }
        full |= !placed;
      };
#pragma unroll
      for (int q = 0; q < kPackEntries; ++q) {
        const int32_t col = poff[kPackEntries * (size_t)p + q];
        if (col < 0) continue;
        const double val = -pval[kPackEntries * (size_t)p + q];
        full |= top_word(val) > kMergeMax;
        if (col < gs) {
          add(col, val);
        } else {
          const int cnt = moff[kMergeStride * (size_t)col + kMergeEntries];
          for (int u = 0; u < cnt; ++u)
            add(mpos[kMergeEntries * (size_t)col + u], -val * mval[kMergeEntries * (size_t)col + u]);
        }
      }
      int cnt = 0;
#pragma unroll
      for (int q = 0; q < kMergeEntries; ++q) {
        cnt += c[q] >= 0;
        full |= top_word(v[q]) > kMergeMax;
        mpos[kMergeEntries * (size_t)p + q] = c[q];
        moff[kMergeStride * (size_t)p + q] = c[q] & (level_window<double>() - 1);
        mval[kMergeEntries * (size_t)p + q] = -v[q];  // (the solve subtracts)
      }
      moff[kMergeStride * (size_t)p + kMergeEntries] = cnt;
      if (full) atomicOr(pflags, kPackMergeFull);
    }
    __syncthreads();  // the level's merged rows are visible to the block
  }
}

// t = the scaled right-hand side with the rows of the own group eliminated
// (as it is when the rows could not be merged), one block per group.
__global__ void __launch_bounds__(256) group_rhs_kernel(int nlev, int r, const int32_t* __restrict__ lvlptr,
                                                        const int32_t* __restrict__ poff,
                                                        const double* __restrict__ pval,
                                                        const double* __restrict__ dinv,
                                                        const int32_t* __restrict__ xrow, const double* __restrict__ x,
                                                        double* t, const uint32_t* __restrict__ pflags) {
  const int l0 = blockIdx.x * r;
  const int l1 = l0 + r < nlev ? l0 + r : nlev;
  const int gs = lvlptr[l0];
  const bool merged = !*pflags;
  for (int l = l0; l < l1; ++l) {
    const int e = lvlptr[l + 1];
    for (int p = lvlptr[l] + (int)threadIdx.x; p < e; p += blockDim.x) {
      double acc = dinv[p] * x[xrow[p]];
      if (merged && l > l0) {
        const int4 c = reinterpret_cast<const int4*>(poff)[p];
        const double* v = pval + kPackEntries * (size_t)p;
        if (c.x >= gs) acc = fma(-v[0], t[c.x], acc);
        if (c.y >= gs) acc = fma(-v[1], t[c.y], acc);
        if (c.z >= gs) acc = fma(-v[2], t[c.z], acc);
        if (c.w >= gs) acc = fma(-v[3], t[c.w], acc);
      }
      t[p] = acc;
    }
    __syncthreads();
  }
}

// The solve of the packed form by T threads, LPR lanes per row: one for real
// rows, two for complex ones (the real and the imaginary part).  A thread has
// up to ROWS rows of a group in registers, loaded D groups ahead (what is wider
// than that goes through memory).  NEAR: every entry is in the ring.
//
// A sub-core of this chip takes one FP64 warp instruction every 64 cycles,
// however few of its lanes are live, and all four together one every 19
// (measured), so what counts is the number of FP64 instructions on the fullest
// sub-core.  A warp therefore runs as many entries as its longest row has --
// one branch to straight-line code, the shorter rows against a zero slot -- and
// not a predicated FMA for every place of the packed form; and a complex row's
// 16 FMAs are spread over two lanes.
//
// Nothing is computed from a row before its group's turn: an operation on what
// was loaded waits for the load (0.36 against 0.18 ms a solve with the values
// negated on arrival).
template <class S, int K>
struct PackedRow {
  int32_t c[K];  // positions (-1: none); of merged rows ring slots, then the count in n
  int32_t n;
  S v[K];
  double x;
  __device__ __forceinline__ void load(const int32_t* off, const S* val, const double* t, size_t p, int lpr, int part) {
    if constexpr (K == kMergeEntries) {
      const int4* o = reinterpret_cast<const int4*>(off + kMergeStride * p);
      const int4 w0 = __ldg(o), w1 = __ldg(o + 1);
      c[0] = w0.x; c[1] = w0.y; c[2] = w0.z; c[3] = w0.w;
      c[4] = w1.x; c[5] = w1.y;
      n = w1.z;
    } else {
      const int4 w = __ldg(reinterpret_cast<const int4*>(off + K * p));
      c[0] = w.x; c[1] = w.y; c[2] = w.z; c[3] = w.w;
    }
    constexpr int PV = 16 / (int)sizeof(S);
    const Pack16<S>* vv = reinterpret_cast<const Pack16<S>*>(val + K * p);
#pragma unroll
    for (int q = 0; q < K / PV; ++q) {
      const Pack16<S> w = vv[q];
#pragma unroll
      for (int u = 0; u < PV; ++u) v[q * PV + u] = w.v[u];
    }
    x = t[lpr * p + part];
  }
};

template <class S, int K, int T, int ROWS, int D, bool NEAR>
__device__ __forceinline__ void packed_solve(int ng, const int32_t* __restrict__ ptr, const int32_t* __restrict__ off,
                                             const S* __restrict__ val, double* t, double* tw) {
  constexpr int kWin = level_window<S>();
  constexpr int LPR = ScalarInfo<S>::cplx ? 2 : 1;
  constexpr int TR = T / LPR;  // rows in step
  constexpr bool kRingSlots = K == kMergeEntries;
  const int tid = (int)threadIdx.x / LPR, part = LPR == 2 ? (int)threadIdx.x & 1 : 0;
  const int wrow = ((int)threadIdx.x & ~31) / LPR;  // the warp's first row
  const int odd = part << 31;
  PackedRow<S, K> row[D][ROWS];
  auto fetch = [&](PackedRow<S, K>(&w)[ROWS], int g) {
    const int b = ptr[g] + tid, e = ptr[g + 1];
#pragma unroll
    for (int u = 0; u < ROWS; ++u)
      if (b + u * TR < e) w[u].load(off, val, t, b + u * TR, LPR, part);
  };
#pragma unroll
  for (int k = 0; k < D; ++k)
    if (k < ng) fetch(row[k], k);
  int b = 0;
  for (int g0 = 0; g0 < ng; g0 += D) {
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const int g = g0 + k;
      if (g >= ng) break;  // uniform
      const int e = ptr[g + 1];
      // a warp's 32 / LPR rows from its own one on; live: the lane has a row
      auto solve = [&](const PackedRow<S, K>& w, int p, bool live) {
        int n = 0;
        if constexpr (kRingSlots) {
          if (live) n = w.n;
        } else {
          if (live) n = w.c[3] >= 0 ? 4 : (w.c[2] >= 0 ? 3 : (w.c[1] >= 0 ? 2 : (w.c[0] >= 0 ? 1 : 0)));
        }
        const int nw = __reduce_max_sync(DIAF_FULL, n);
        double acc = w.x;
        auto run = [&](auto count) {
          constexpr int Q = decltype(count)::value;
          const double* src[Q];
#pragma unroll
          for (int q = 0; q < Q; ++q) {
            const bool has = q < n;
            if (kRingSlots) src[q] = tw + (has ? w.c[q] : kWin);
            else if (NEAR) src[q] = tw + LPR * (has ? w.c[q] & (kWin - 1) : kWin);
            else src[q] = !has || w.c[q] >= e - kWin ? tw + LPR * (has ? w.c[q] & (kWin - 1) : kWin)
                                                     : t + (size_t)LPR * w.c[q];
          }
          if constexpr (LPR == 1) {
            double tv[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) tv[q] = *src[q];
#pragma unroll
            for (int q = 0; q < Q; ++q) acc = fma(-w.v[q], tv[q], acc);
          } else {  // re: (acc - v.re t.re) + v.im t.im; im: (acc - v.re t.im) - v.im t.re
            double t0[Q], t1[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) {
              t0[q] = src[q][part];
              t1[q] = src[q][1 - part];
            }
#pragma unroll
            for (int q = 0; q < Q; ++q) {
              const double im = __hiloint2double(__double2hiint(w.v[q].im) ^ odd, __double2loint(w.v[q].im));
              acc = fma(im, t1[q], fma(-w.v[q].re, t0[q], acc));
            }
          }
        };
        if (nw == 2) run(std::integral_constant<int, 2>());
        else if (nw == 3) run(std::integral_constant<int, 3>());
        else if (nw == 4) run(std::integral_constant<int, 4>());
        else if (nw == 1) run(std::integral_constant<int, 1>());
        else if (K > 4 && nw == 5) run(std::integral_constant<int, K < 5 ? K : 5>());
        else if (K > 4 && nw == 6) run(std::integral_constant<int, K < 6 ? K : 6>());
        if (live) {
          t[(size_t)LPR * p + part] = acc;
          tw[LPR * (p & (kWin - 1)) + part] = acc;
        }
      };
#pragma unroll
      for (int u = 0; u < ROWS; ++u)
        if (b + wrow + u * TR < e) solve(row[k][u], b + tid + u * TR, b + tid + u * TR < e);
      for (int p0 = b + wrow + ROWS * TR; p0 < e; p0 += TR) {
        const int p = p0 + tid - wrow;
        PackedRow<S, K> w;
        if (p < e) w.load(off, val, t, p, LPR, part);
        solve(w, p, p < e);
      }
      if (g + D < ng) fetch(row[k], g + D);
      b = e;
      __syncthreads();
    }
  }
}

// One block of T threads, ROWS rows of a group in a thread's registers.
// MERGED: groups of r levels.
template <class S, int T, int ROWS, int D, bool MERGED>
__global__ void __launch_bounds__(T, 1)
    trsv_packed_kernel(int nlev, int r, const int32_t* __restrict__ lvlptr, const int32_t* __restrict__ poff,
                       const S* __restrict__ pval, const int32_t* __restrict__ moff, const double* __restrict__ mval,
                       const uint32_t* __restrict__ pflags, double* t) {
  extern __shared__ __align__(16) unsigned char level_ring[];
  double* tw = reinterpret_cast<double*>(level_ring);
  if (threadIdx.x < 2) tw[level_window<double>() + threadIdx.x] = 0.0;  // the zero slot
  __shared__ int32_t sptr[kLevelPtrSmem + 1];
  const uint32_t fl = *pflags;
  const bool merged = MERGED && !fl;
  const int step = merged ? r : 1;
  const int ng = (nlev + step - 1) / step;
  const bool in_smem = ng <= kLevelPtrSmem;
  if (in_smem)
    for (int i = threadIdx.x; i <= ng; i += T) sptr[i] = lvlptr[i * step < nlev ? i * step : nlev];
  __syncthreads();
  if constexpr (MERGED) {
    if (merged && in_smem) {
      packed_solve<double, kMergeEntries, T, ROWS, D, true>(ng, sptr, moff, mval, t, tw);
      return;
    }
  }
  // (the host groups levels only where their pointers fit in shared memory)
  const int32_t* ptr = in_smem ? sptr : lvlptr;
  if (!(fl & kPackFar)) packed_solve<S, kPackEntries, T, ROWS, D, true>(ng, ptr, poff, pval, t, tw);
  else packed_solve<S, kPackEntries, T, ROWS, 1, false>(ng, ptr, poff, pval, t, tw);
}

}  // namespace

int level_group(bool cplx, int maxrow, int nlev, const int32_t* lvlptr, int* maxg) {
  *maxg = 0;
  if (maxrow > kPackEntries || nlev <= 0) return 0;
  for (int r = cplx ? 1 : 4; r >= 1; r >>= 1) {
    int w = 0;
    for (int l = 0; l < nlev; l += r) {
      const int n = lvlptr[l + r < nlev ? l + r : nlev] - lvlptr[l];
      if (n > w) w = n;
    }
    if ((w <= kGroupRows && nlev <= r * kLevelPtrSmem) || r == 1) {
      *maxg = w;
      return r;
    }
  }
  return 0;
}

cudaError_t level_place(int n, bool cplx, const int32_t* lev, const int32_t* rank, const int32_t* rcnt, int32_t* pos,
                        int32_t* work, LevelCsr& L, cudaStream_t s) {
  if (n <= 0) return cudaMemsetAsync(L.rowptr, 0, sizeof(int32_t), s);
  int32_t* len = work;
  int32_t* bs = work + n;
  const bool rows = L.r == 0 || cplx;  // the rows' pointers are needed
  level_place_kernel<<<ceil_div(n, 256), 256, 0, s>>>(n, lev, rank, rcnt, L.lvlptr, pos, L.xrow, len,
                                                      rows ? nullptr : L.poff, (double*)L.pval);
  DIAF_COUNT_LAUNCH();
  return rows ? exclusive_scan_i32(len, L.rowptr, n, bs, s) : cudaGetLastError();
}

cudaError_t level_fill(int n, bool cplx, const int32_t* cp, const int32_t* ri, const void* v, const int32_t* dpos,
                       const int32_t* slot, const int32_t* pos, const int32_t* lev, LevelCsr& L, uint32_t* zflag,
                       cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int blocks = (int)(((int64_t)n * kConvLanes + 255) / 256);
  if (L.r > 0) {
    cudaError_t e = cudaMemsetAsync(L.pflags, 0, sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
  }
  if (cplx) {
    level_fill_kernel<Cx<double>><<<blocks, 256, 0, s>>>(n, cp, ri, (const Cx<double>*)v, dpos, slot, pos, L.rowptr,
                                                          L.colidx, (Cx<double>*)L.vals, (Cx<double>*)L.dinv, zflag);
    DIAF_COUNT_LAUNCH();
    if (L.r > 0) {
      pack_rows_kernel<<<L.nlev < 4096 ? L.nlev : 4096, 128, 0, s>>>(L.nlev, L.lvlptr, L.rowptr, L.colidx,
                                                                     (const Cx<double>*)L.vals, L.poff,
                                                                     (Cx<double>*)L.pval, L.pflags);
      DIAF_COUNT_LAUNCH();
    }
  } else if (L.r > 0) {
    packed_fill_kernel<<<blocks, 256, 0, s>>>(n, cp, ri, (const double*)v, dpos, slot, pos, lev, L.lvlptr, L.r, L.nlev,
                                              L.poff, (double*)L.pval, (double*)L.dinv, zflag, L.pflags);
    DIAF_COUNT_LAUNCH();
    if (L.r > 1) {
      merge_kernel<<<ceil_div(L.nlev, L.r), 256, 0, s>>>(L.nlev, L.r, L.lvlptr, L.poff, (const double*)L.pval, L.mpos,
                                                         L.moff, L.mval, L.pflags);
      DIAF_COUNT_LAUNCH();
    }
  } else {
    level_fill_kernel<double><<<blocks, 256, 0, s>>>(n, cp, ri, (const double*)v, dpos, slot, pos, L.rowptr, L.colidx,
                                                      (double*)L.vals, (double*)L.dinv, zflag);
    DIAF_COUNT_LAUNCH();
  }
  return cudaGetLastError();
}

cudaError_t remap_columns(int64_t nnz, const int32_t* pos, const int32_t* cin, int32_t* cout, cudaStream_t s) {
  if (nnz <= 0) return cudaSuccess;
  int blocks = (int)((nnz + 255) / 256);
  if (blocks > 4096) blocks = 4096;
  remap_cols_kernel<<<blocks, 256, 0, s>>>(nnz, pos, cin, cout);
  DIAF_COUNT_LAUNCH();
  return cudaGetLastError();
}

template <class S, int T, int ROWS, int D, bool MERGED>
static cudaError_t trsv_packed_t(const LevelCsr& L, void* t, cudaStream_t s) {
  constexpr size_t ring = sizeof(S) * level_window<S>() + 16;  // and the zero slot
  static std::atomic<uint64_t> configured{0};  // the attribute is per device: one bit each
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = 1ull << (dev & 63);
  if (dev > 63 || !(configured.load() & bit)) {
    e = cudaFuncSetAttribute(trsv_packed_kernel<S, T, ROWS, D, MERGED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)ring);
    if (e != cudaSuccess) return e;
    configured.fetch_or(bit);
  }
  trsv_packed_kernel<S, T, ROWS, D, MERGED><<<1, T, ring, s>>>(L.nlev, L.r, L.lvlptr, L.poff, (const S*)L.pval, L.moff,
                                                         L.mval, L.pflags, (double*)t);
  DIAF_COUNT_LAUNCH();
  return cudaGetLastError();
}

template <class S, bool MERGED>
static cudaError_t trsv_packed(const LevelCsr& L, const void* x, void* t, cudaStream_t s) {
  if constexpr (MERGED)
    group_rhs_kernel<<<ceil_div(L.nlev, L.r), 256, 0, s>>>(L.nlev, L.r, L.lvlptr, L.poff, (const double*)L.pval,
                                                           (const double*)L.dinv, L.xrow, (const double*)x,
                                                           (double*)t, L.pflags);
  else
    scale_rhs_kernel<S><<<ceil_div(L.n, 256), 256, 0, s>>>(L.n, (const S*)L.dinv, L.xrow, (const S*)x, (S*)t);
  DIAF_COUNT_LAUNCH();
  // (64 registers a thread, as 1,024 threads would have, spill: more rows each instead)
  if constexpr (ScalarInfo<S>::cplx) {
    if (L.maxg <= 128) return trsv_packed_t<S, 256, 1, 4, MERGED>(L, t, s);
    if (L.maxg <= 256) return trsv_packed_t<S, 512, 1, 2, MERGED>(L, t, s);
    return trsv_packed_t<S, 512, 2, 1, MERGED>(L, t, s);
  } else {
    if (L.maxg <= 256) return trsv_packed_t<S, 256, 1, 4, MERGED>(L, t, s);
    if (L.maxg <= 512) return trsv_packed_t<S, 512, 1, 2, MERGED>(L, t, s);
    return trsv_packed_t<S, 512, 2, 2, MERGED>(L, t, s);
  }
}

template <class S>
static cudaError_t trsv_levels_perm_t(const LevelCsr& L, const void* x, void* t, bool warm, cudaStream_t s) {
  constexpr size_t ring = sizeof(S) * level_window<S>();
  static int configured_device = -1;  // the attribute is per device
  int dev = 0;
  cudaGetDevice(&dev);
  if (configured_device != dev) {
    cudaError_t e = cudaFuncSetAttribute(trsv_levels_perm_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)ring);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(trsv_levels_deep_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ring);
    if (e != cudaSuccess) return e;
    configured_device = dev;
  }
  scale_rhs_kernel<S><<<ceil_div(L.n, 256), 256, 0, s>>>(L.n, (const S*)L.dinv, L.xrow, (const S*)x, (S*)t);
  DIAF_COUNT_LAUNCH();
  if (L.maxw <= kDeepThreads)
    trsv_levels_deep_kernel<S><<<1, kDeepThreads, ring, s>>>(L.nlev, L.lvlptr, L.rowptr, L.colidx,
                                                             (const S*)L.vals, (S*)t, warm ? 1 : 0);
  else
    trsv_levels_perm_kernel<S><<<1, kLevelThreads, ring, s>>>(L.nlev, L.lvlptr, L.rowptr, L.colidx,
                                                              (const S*)L.vals, (S*)t, warm ? 1 : 0);
  DIAF_COUNT_LAUNCH();
  return cudaGetLastError();
}

cudaError_t trsv_levels_perm(const LevelCsr& L, bool cplx, const void* x, void* t, cudaStream_t s, bool warm) {
  if (L.n <= 0) return cudaSuccess;
  if (L.r > 1) return trsv_packed<double, true>(L, x, t, s);
  if (L.r == 1) return cplx ? trsv_packed<Cx<double>, false>(L, x, t, s) : trsv_packed<double, false>(L, x, t, s);
  return cplx ? trsv_levels_perm_t<Cx<double>>(L, x, t, warm, s) : trsv_levels_perm_t<double>(L, x, t, warm, s);
}

cudaError_t csc_to_csr(int n, int64_t nnz, const int32_t* cp, const int32_t* ri, const void* v, bool cplx,
                       int32_t* rowptr, int32_t* colidx, void* vals, int32_t* work, cudaStream_t s) {
  if (cplx)
    return csc_to_csr_t<Cx<double>>(n, nnz, cp, ri, (const Cx<double>*)v, rowptr, colidx, (Cx<double>*)vals, work, s);
  return csc_to_csr_t<double>(n, nnz, cp, ri, (const double*)v, rowptr, colidx, (double*)vals, work, s);
}

cudaError_t csr_spmv(const Csr& M, bool cplx, const void* x, void* y, cudaStream_t s) {
  if (M.n <= 0) return cudaSuccess;
  constexpr int G = 4;
  int threads = 256;
  int blocks = ceil_div(M.n * G, threads);
  if (cplx)
    spmv_kernel<Cx<double>, G><<<blocks, threads, 0, s>>>(M.n, M.rowptr, M.colidx, (const Cx<double>*)M.vals,
                                                          (const Cx<double>*)x, (Cx<double>*)y);
  else
    spmv_kernel<double, G><<<blocks, threads, 0, s>>>(M.n, M.rowptr, M.colidx, (const double*)M.vals,
                                                      (const double*)x, (double*)y);
  DIAF_COUNT_LAUNCH();
  return cudaGetLastError();
}


