// Linear solves in A = I + alpha L (the matrix of the grounded pivot system of
// Algorithm 1, and of the CG ground truth of Sec. 6.1), and in the Laplacian
// L of a connected G itself (the pivot column of L^+ that the electrical-
// closeness algorithm of Sec. 3 needs): A = sigma I + alpha L, sigma 1 or 0.
//
// Mixed precision: the outer loop is iterative refinement in FP64
// (r = b - A x with FP64 x and FP64 arithmetic, x += correction); the
// correction solves A d = r / ||r|| with Jacobi-preconditioned CG in FP32.
// Several right-hand sides run side by side (column j of an [m][n] block),
// each with its own CG scalars; reductions are two-pass and fixed-order, so
// results do not depend on scheduling.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "fc_internal.cuh"

namespace cgr = cooperative_groups;

namespace fcx {

constexpr int SV_T = 256;

// Block-wide sum of two doubles (warp shuffles, then one warp); the result
// is valid in thread 0.
__device__ __forceinline__ void block_sum2(double& a, double& b) {
  __shared__ double wa[SV_T / 32], wb[SV_T / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  if ((threadIdx.x & 31) == 0) {
    wa[threadIdx.x >> 5] = a;
    wb[threadIdx.x >> 5] = b;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    a = 0.0;
    b = 0.0;
    for (int w = 0; w < SV_T / 32; ++w) {
      a += wa[w];
      b += wb[w];
    }
  }
}

__global__ void k_colsum(const double* __restrict__ part, int nb, double* __restrict__ out) {
  __shared__ double red[SV_T];
  const int j = blockIdx.x;
  double s = 0.0;
  for (int i = threadIdx.x; i < nb; i += SV_T) s += part[(size_t)j * nb + i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int k = SV_T / 2; k > 0; k >>= 1) {
    if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[j] = red[0];
}

// ---- FP32 inner PCG ---------------------------------------------------------
struct Inner {
  float* r;   // residual of the correction system
  float* p;
  float* q;
  float* d;   // correction
  double* scal;  // per column: [0] rz, [1] pq, [2] rz_new, [3] rr, [4] scale, [5] active
};

// r32 = r64 * inv_scale; d = 0; p = z = r32 / diag; partial r.z and r.r
__global__ void k_inner_init(int32_t n, const double* __restrict__ r64, const float* __restrict__ prec,
                             const double* __restrict__ scal, Inner in, double* __restrict__ prz,
                             double* __restrict__ prr, int nb) {
  const int j = blockIdx.y;
  const size_t off = (size_t)j * n;
  const double sc = scal[j * 8 + 4];
  float rzf = 0.0f, rrf = 0.0f;  // per-thread partials in FP32, then FP64 across threads
  for (int64_t v = (int64_t)blockIdx.x * SV_T + threadIdx.x; v < n; v += (int64_t)gridDim.x * SV_T) {
    const float rv = (float)(r64[off + v] * sc);
    const float z = prec ? rv * prec[v] : rv;
    in.r[off + v] = rv;
    in.p[off + v] = z;
    in.d[off + v] = 0.0f;
    rzf = fmaf(rv, z, rzf);
    rrf = fmaf(rv, rv, rrf);
  }
  double rz = rzf, rr = rrf;
  block_sum2(rz, rr);
  if (threadIdx.x == 0) {
    prz[(size_t)j * nb + blockIdx.x] = rz;
    prr[(size_t)j * nb + blockIdx.x] = rr;
  }
}

// x += (1/scale) d (FP64), only for active columns
__global__ void k_correct(int32_t n, const double* __restrict__ scal, const float* __restrict__ d,
                          double* __restrict__ x) {
  const int j = blockIdx.y;
  const double* sc = scal + j * 8;
  if (sc[5] == 0.0) return;
  const double f = 1.0 / sc[4];  // one division per thread: GB300's FP64 rate is low (n = 2.1M: 90 us
  // with a division per entry)
  const size_t off = (size_t)j * n;
  for (int64_t v = (int64_t)blockIdx.x * SV_T + threadIdx.x; v < n; v += (int64_t)gridDim.x * SV_T)
    x[off + v] += (double)d[off + v] * f;
}

// the FP32 diagonal and its reciprocal (the Jacobi preconditioner, applied
// as a product)
__global__ void k_diag32(int32_t n, const double* __restrict__ dw, double sigma, double alpha,
                         float* __restrict__ diag32, float* __restrict__ inv32) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n) {
    const double d = sigma + alpha * dw[v];
    diag32[v] = (float)d;
    inv32[v] = (float)(1.0 / d);
  }
}

__global__ void k_fill(int64_t len, double val, double* __restrict__ a) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < len) a[i] = val;
}

// x over V' (n+1 entries, x[n] = x(u*) = 0 on entry) -> mean-zero gauge
__global__ void k_shift(int64_t len, const double* __restrict__ sum, double* __restrict__ x) {
  const double mean = *sum / (double)len;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x)
    x[i] -= mean;
}

// *any = 1 where an entry differs from zero
__global__ void k_any_nonzero(int64_t len, const double* __restrict__ x, uint32_t* __restrict__ any) {
  bool nz = false;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x)
    nz |= x[i] != 0.0;
  if (__syncthreads_or(nz) && threadIdx.x == 0) atomicOr(any, 1u);
}

__global__ void k_partial_sum(int64_t len, const double* __restrict__ a, double* __restrict__ part) {
  __shared__ double red[SV_T];
  const int64_t i = (int64_t)blockIdx.x * SV_T + threadIdx.x;
  red[threadIdx.x] = i < len ? a[i] : 0.0;
  __syncthreads();
  for (int s = SV_T / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}


// Singular systems (sigma = 0, L of a connected graph): the residual's
// component along 1 lies in L's kernel, where CG cannot reduce it; rounding
// in the FP64 residual leaves a little there, so each refinement step
// projects it out.  Element (v, j) of the columns at v sv + j sj (column-major
// or interleaved); blockIdx.y = j, fixed-order partial sums of the column per
// block (one block per column took 0.4 ms for one column of n = 2^18, most of
// a Laplacian solve).
__global__ void __launch_bounds__(SV_T) k_col_part(int32_t n, const double* __restrict__ in, int64_t sv, int64_t sj,
                                                   double* __restrict__ part, int nb) {
  const double* x = in + blockIdx.y * sj;
  double s = 0.0, unused = 0.0;
  for (int64_t v = (int64_t)blockIdx.x * SV_T + threadIdx.x; v < n; v += (int64_t)gridDim.x * SV_T) s += x[v * sv];
  block_sum2(s, unused);
  if (threadIdx.x == 0) part[(size_t)blockIdx.y * nb + blockIdx.x] = s;
}

// out = in - sum_j / n; partial sums of squares of out (part may be null)
__global__ void __launch_bounds__(SV_T) k_col_shift(int32_t n, const double* in, int64_t sv, int64_t sj,
                                                    const double* __restrict__ sums, double* out,
                                                    double* __restrict__ part, int nb) {
  const double mean = sums[blockIdx.y] / (double)n;
  double q = 0.0, unused = 0.0;
  for (int64_t v = (int64_t)blockIdx.x * SV_T + threadIdx.x; v < n; v += (int64_t)gridDim.x * SV_T) {
    const double x = in[v * sv + blockIdx.y * sj] - mean;
    out[v * sv + blockIdx.y * sj] = x;
    q += x * x;
  }
  if (part == nullptr) return;
  block_sum2(q, unused);
  if (threadIdx.x == 0) part[(size_t)blockIdx.y * nb + blockIdx.x] = q;
}

// Both in one launch for columns of up to COL_ONE entries, a block per column:
// out = in - mean, sums of squares of out (sq may be null).
constexpr int COL_ONE = 8192;
__global__ void __launch_bounds__(SV_T) k_col_center(int32_t n, const double* in, int64_t sv, int64_t sj, double* out,
                                                     double* __restrict__ sq) {
  __shared__ double mean;
  const int64_t off = blockIdx.x * sj;
  double s = 0.0, unused = 0.0;
  for (int64_t v = threadIdx.x; v < n; v += SV_T) s += in[v * sv + off];
  block_sum2(s, unused);
  if (threadIdx.x == 0) mean = s / (double)n;
  __syncthreads();
  double q = 0.0;
  for (int64_t v = threadIdx.x; v < n; v += SV_T) {
    const double x = in[v * sv + off] - mean;
    out[v * sv + off] = x;
    q += x * x;
  }
  block_sum2(q, unused);
  if (sq && threadIdx.x == 0) sq[blockIdx.x] = q;
}

// out = in - mean for m columns of n entries (element (v, j) at v sv + j sj; in
// place when out is in); sq (or null): their sums of squares.  part: [m][nb + 1].
// One launch for short columns, else four over many blocks.  Measured on GB300
// (whole Laplacian solves of one column, four launches -> one): complete graph of
// 600 495 -> 455 us, ER n = 6000 743 -> 711; n = 12,000 is even (735).
static fc_status center_columns(int32_t n, int m, const double* in, int64_t sv, int64_t sj, double* out, double* sq,
                                double* part, int nb, cudaStream_t st) {
  if (n <= COL_ONE) {
    k_col_center<<<m, SV_T, 0, st>>>(n, in, sv, sj, out, sq);
    FC_LAUNCHED();
    return FC_OK;
  }
  double* sums = part + (size_t)m * nb;
  k_col_part<<<dim3(nb, m), SV_T, 0, st>>>(n, in, sv, sj, part, nb);
  FC_LAUNCHED();
  k_colsum<<<m, SV_T, 0, st>>>(part, nb, sums);
  FC_LAUNCHED();
  k_col_shift<<<dim3(nb, m), SV_T, 0, st>>>(n, in, sv, sj, sums, out, sq ? part : nullptr, nb);
  FC_LAUNCHED();
  if (sq) {
    k_colsum<<<m, SV_T, 0, st>>>(part, nb, sq);
    FC_LAUNCHED();
  }
  return FC_OK;
}

// ---------------------------------------------------------------------------
// One right-hand side.
//
// Sums over rows, s_v = sum_j w_vj x_j, in edge tiles: tile t holds the
// entries [t TL, (t+1) TL) of the CSR arrays and is one warp, TL_E
// consecutive entries per lane, whatever the rows.  A row of a few thousand
// entries (the hubs of a scale-free graph) is spread over many lanes and
// warps instead of serialising one group of lanes, and every lane issues TL_E
// independent gathers.  Within a tile a segmented scan over the lanes' last
// rows (keys nondecreasing) joins rows that cross lanes; a row that crosses
// tiles leaves one partial per tile (tail[t0] in the tile where it starts,
// head[t] in each later tile) and is summed from them in tile order.  Tiles
// need no block barrier, so the warps of a block hide each other's memory
// latency.  Every addition has a fixed place, so results do not depend on
// scheduling.
// ---------------------------------------------------------------------------
constexpr int TL_T = 32;              // lanes per tile (one warp)
constexpr int TL_E = 8;               // entries per lane
constexpr int TL = TL_T * TL_E;       // entries per tile
constexpr int TL_RCAP = TL + 2;       // row offsets staged in shared memory (general tiles)
constexpr int TL_W = SV_T / 32;       // tiles in flight per block

// row0[t] / row1[t]: the rows holding the first / last entry of tile t (the
// largest v with rowptr[v] <= e)
__global__ void k_tile_rows(int32_t n, int64_t nnz, const int64_t* __restrict__ rowptr, int64_t ntiles,
                            int32_t* __restrict__ row0, int32_t* __restrict__ row1) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 2 * ntiles) return;
  const int64_t t = i >> 1;
  const int64_t e = (i & 1) ? std::min<int64_t>((t + 1) * TL, nnz) - 1 : t * TL;
  int32_t lo = 0, hi = n - 1;
  while (lo < hi) {
    const int32_t mid = lo + (hi - lo + 1) / 2;
    if (rowptr[mid] <= e) lo = mid;
    else hi = mid - 1;
  }
  ((i & 1) ? row1 : row0)[t] = lo;
}

// Per-thread tile metadata, one word per thread, fixed for the whole solve:
//   bit j (1..TL_E-1)  entry j of the thread starts a new row
//   bit TM_EL          the thread's last row ends at its last entry
//   bits TM_RF..       the row of its first entry, relative to row0[t]
//   TM_BEFORE          the tile's first row began in an earlier tile
//   TM_GENERAL         the tile has empty rows between its first and last
//                      row: walked through the row offsets instead
constexpr uint32_t TM_EL = 1u << TL_E;
constexpr int TM_RF = TL_E + 1;
constexpr uint32_t TM_RF_MASK = 0xFFFu;
constexpr uint32_t TM_BEFORE = 1u << 29;
constexpr uint32_t TM_GENERAL = 1u << 30;

__global__ void __launch_bounds__(SV_T) k_tile_meta(int64_t nnz, const int64_t* __restrict__ rowptr, int64_t ntiles,
                                                    const int32_t* __restrict__ row0,
                                                    const int32_t* __restrict__ row1, uint32_t* __restrict__ meta) {
  const int lane = threadIdx.x & 31;
  for (int64_t t = (int64_t)blockIdx.x * TL_W + (threadIdx.x >> 5); t < ntiles; t += (int64_t)gridDim.x * TL_W) {
    const int64_t E0 = t * TL;
    const int ne = (int)std::min<int64_t>(TL, nnz - E0);
    const int32_t rs = row0[t];
    const int nr = row1[t] - rs + 1;
    int empty = 0;
    for (int i = 1 + lane; i < nr; i += TL_T) empty |= rowptr[rs + i + 1] == rowptr[rs + i];
    const bool general = __any_sync(0xffffffffu, empty) != 0;
    uint32_t mw = (general ? TM_GENERAL : 0u) | (rowptr[rs] < E0 ? TM_BEFORE : 0u);
    const int le0 = lane * TL_E;
    const int cnt = ne - le0 >= TL_E ? TL_E : (ne - le0 > 0 ? ne - le0 : 0);
    if (!general && cnt > 0) {
      int lo = 0, hi = nr - 1;  // the row holding entry le0
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (rowptr[rs + mid] - E0 <= le0) lo = mid;
        else hi = mid - 1;
      }
      mw |= (uint32_t)lo << TM_RF;
      int cur = lo;
      int64_t nxt = rowptr[rs + cur + 1] - E0;
      for (int j = 1; j < cnt; ++j)
        if (nxt == le0 + j) {  // no empty rows here: one row per boundary
          mw |= 1u << j;
          ++cur;
          nxt = rowptr[rs + cur + 1] - E0;
        }
      if (nxt == le0 + cnt) mw |= TM_EL;
    }
    meta[t * TL_T + lane] = mw;
  }
}

struct TileSmem {
  int32_t off[TL_W][TL_RCAP];  // rowptr[row0 + i] - t TL (general tiles), one row per warp
};

template <typename V>
struct TileArgs {
  int64_t nnz;
  const int64_t* rowptr;
  const int32_t* colidx;
  const float* w;
  const int32_t* row0;
  const int32_t* row1;
  const uint32_t* meta;  // [tiles][TL_T] from k_tile_meta
  const uint32_t* span;  // bit v: row v is empty or crosses tiles (s[v] not written)
  V* s;     // rows inside one tile
  V* head;  // [tiles] partial of the tile's first row if it began earlier
  V* tail;  // [tiles] partial of the tile's last row if it began here and goes on
  bool vec; // colidx / w 16-byte aligned: vector loads for full tiles
};

// What a lane needs of one tile before its gathers, loaded one tile ahead.
struct TileIn {
  int32_t col[TL_E];
  uint32_t mw;
  int32_t rs;
};

// The matrix is streamed with an evict-first hint, so that the vectors stay in L2
// across an iteration: one column on a weighted 2.1M-vertex grid (matrix 67 MB,
// vectors 59 MB, L2 129 MB) 6.82 -> 6.04 ms a solve.
template <typename V>
__device__ __forceinline__ void tile_load(const TileArgs<V>& a, int64_t t, TileIn& ti) {
  const int lane = threadIdx.x & 31;
  const int64_t E0 = t * TL;
  const int ne = (int)std::min<int64_t>(TL, a.nnz - E0);
  const int le0 = lane * TL_E;
  const int cnt = ne - le0 >= TL_E ? TL_E : (ne - le0 > 0 ? ne - le0 : 0);
  ti.rs = a.row0[t];
  ti.mw = __ldcs(a.meta + t * TL_T + lane);
  if (a.vec && ne == TL) {
    const int4* c4 = reinterpret_cast<const int4*>(a.colidx + E0 + le0);
    const int4 c0 = __ldcs(c4), c1 = __ldcs(c4 + 1);
    ti.col[0] = c0.x; ti.col[1] = c0.y; ti.col[2] = c0.z; ti.col[3] = c0.w;
    ti.col[4] = c1.x; ti.col[5] = c1.y; ti.col[6] = c1.z; ti.col[7] = c1.w;
  } else {
#pragma unroll
    for (int j = 0; j < TL_E; ++j) ti.col[j] = j < cnt ? a.colidx[E0 + le0 + j] : 0;
  }
}

// Folded form (FP32 inner CG): a tile finishes q_v = diag_v p_v - alpha s_v
// of every row that lies inside it, and every tile adds its rows' terms of
// p.q to a per-lane partial: p_v q_v for rows inside, and for a row that
// crosses tiles the linear pieces p_v diag_v p_v (in the tile where it
// starts) and -alpha p_v times the tile's partial (in every tile it touches).
struct Fold {
  const float* diag;
  float alpha;
  float* q;
};

// One tile of s = W x, by one whole warp, from its loaded indices.
template <typename V, bool FOLD = false>
__device__ void tile_finish(const TileArgs<V>& a, const V* __restrict__ x, int64_t t, const TileIn& ti,
                            int32_t* __restrict__ soff, const Fold& fo = Fold{}, float* pq = nullptr) {
  // a row's sum is complete: store it, or (folded) finish q and p.q
  auto put_row = [&](int32_t v, V sv) {
    if (FOLD) {
      const float pv = (float)x[v];
      const float qv = pv * fo.diag[v] - fo.alpha * (float)sv;
      fo.q[v] = qv;
      *pq = fmaf(pv, qv, *pq);
    } else {
      a.s[v] = sv;
    }
  };
  const int lane = threadIdx.x & 31;
  const int64_t E0 = t * TL;
  const int ne = (int)std::min<int64_t>(TL, a.nnz - E0);
  const int32_t rs = ti.rs;
  const uint32_t mw = ti.mw;
  const int le0 = lane * TL_E;
  const int cnt = ne - le0 >= TL_E ? TL_E : (ne - le0 > 0 ? ne - le0 : 0);
  float wt[TL_E];
  if (a.w && a.vec && ne == TL) {
    const float4* w4 = reinterpret_cast<const float4*>(a.w + E0 + le0);
    const float4 w0 = __ldcs(w4), w1 = __ldcs(w4 + 1);
    wt[0] = w0.x; wt[1] = w0.y; wt[2] = w0.z; wt[3] = w0.w;
    wt[4] = w1.x; wt[5] = w1.y; wt[6] = w1.z; wt[7] = w1.w;
  } else {
#pragma unroll
    for (int j = 0; j < TL_E; ++j) wt[j] = j < cnt ? (a.w ? a.w[E0 + le0 + j] : 1.0f) : 0.0f;
  }
  V prod[TL_E];
#pragma unroll
  for (int j = 0; j < TL_E; ++j) prod[j] = j < cnt ? (V)wt[j] * x[ti.col[j]] : (V)0;
  // walk this thread's entries: rf / pf its first row and partial, rl / pl
  // its last; rows that start and end inside the thread are written here
  int32_t rf = 0, rl = INT32_MAX;
  V pf = 0, pl = 0;
  bool ef = false, el = false;
  const bool before = (mw & TM_BEFORE) != 0;
  if (!(mw & TM_GENERAL)) {  // uniform over the tile
    if (cnt > 0) {
      rf = (int32_t)((mw >> TM_RF) & TM_RF_MASK);
      int cur = rf;
      V acc = 0;
      bool first = true;
#pragma unroll
      for (int j = 0; j < TL_E; ++j) {
        if (j < cnt) {
          if (j > 0 && ((mw >> j) & 1u)) {  // entry j starts row cur + 1
            if (first) {
              pf = acc;
              ef = true;
              first = false;
            } else {
              put_row(rs + cur, acc);
            }
            acc = 0;
            ++cur;
          }
          acc += prod[j];
        }
      }
      rl = cur;
      pl = acc;
      el = (mw & TM_EL) != 0;
      if (first) {
        pf = acc;
        ef = el;
      }
    }
  } else {
    const int nr = a.row1[t] - rs + 1;  // rows touching the tile, empty ones included
    const bool use_sm = nr + 1 <= TL_RCAP;
    if (use_sm)
      for (int i = lane; i <= nr; i += TL_T) soff[i] = (int32_t)(a.rowptr[rs + i] - E0);
    __syncwarp();
    auto off = [&](int i) -> int32_t { return use_sm ? soff[i] : (int32_t)(a.rowptr[rs + i] - E0); };
    if (cnt > 0) {
      int lo = 0, hi = nr - 1;  // the row holding entry le0
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (off(mid) <= le0) lo = mid;
        else hi = mid - 1;
      }
      rf = lo;
      int cur = lo;
      int32_t beg = off(cur), nxt = off(cur + 1);
      V acc = 0;
      bool first = true;
#pragma unroll
      for (int j = 0; j < TL_E; ++j) {
        if (j < cnt) {
          while (nxt <= le0 + j) {  // row cur ended before this entry
            if (first) {
              pf = acc;
              ef = true;
              first = false;
            } else if (beg < nxt) {
              put_row(rs + cur, acc);
            }
            acc = 0;
            ++cur;
            beg = nxt;
            nxt = off(cur + 1);
          }
          acc += prod[j];
        }
      }
      rl = cur;
      pl = acc;
      el = nxt <= le0 + cnt;
      if (first) {
        pf = acc;
        ef = el;
      }
    }
  }
  // segmented inclusive scan of pl over the lanes, keyed by rl
  V S = pl;
  int32_t key = rl;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const V so = __shfl_up_sync(0xffffffffu, S, d);
    const int32_t ko = __shfl_up_sync(0xffffffffu, key, d);
    if (lane >= d && ko == key) S += so;
  }
  const V Sp = __shfl_up_sync(0xffffffffu, S, 1);  // the previous lane's, for its row
  const int32_t kp = __shfl_up_sync(0xffffffffu, key, 1);
  if (cnt > 0) {
    if (ef) {
      const V tot = (lane > 0 && kp == rf ? Sp : (V)0) + pf;
      if (rf == 0 && before) {
        a.head[t] = tot;
        if (FOLD) *pq = fmaf(-fo.alpha * (float)x[rs], (float)tot, *pq);
      } else {
        put_row(rs + rf, tot);
      }
    }
    if (rl != rf && el) put_row(rs + rl, pl);
    if (le0 + cnt == ne && !el) {  // the tile's last row goes on into the next tile
      if (rl == 0 && before) {
        a.head[t] = S;
        if (FOLD) *pq = fmaf(-fo.alpha * (float)x[rs], (float)S, *pq);
      } else {
        a.tail[t] = S;
        if (FOLD) {
          const int32_t v = rs + rl;
          const float pv = (float)x[v];
          *pq = fmaf(pv, pv * fo.diag[v] - fo.alpha * (float)S, *pq);
        }
      }
    }
  }
  __syncwarp();
}

// The tiles t0, t0 + stride, ... of one warp, each tile's indices loaded
// while the previous tile is summed.
template <typename V, bool FOLD = false>
__device__ __forceinline__ void tile_loop(const TileArgs<V>& a, const V* __restrict__ x, int64_t ntiles, int64_t t0,
                                          int64_t stride, int32_t* __restrict__ soff, const Fold& fo = Fold{},
                                          float* pq = nullptr) {
  TileIn cur, nxt;
  if (t0 < ntiles) tile_load(a, t0, cur);
  for (int64_t t = t0; t < ntiles; t += stride) {
    if (t + stride < ntiles) tile_load(a, t + stride, nxt);
    tile_finish<V, FOLD>(a, x, t, cur, soff, fo, pq);
    cur = nxt;
  }
}

// s_v of a row marked in the span bitmap: 0 if empty, else the sum of its
// tile partials in tile order
template <typename V>
__device__ __forceinline__ V row_total_span(const TileArgs<V>& a, int64_t v) {
  const int64_t e0 = a.rowptr[v], e1 = a.rowptr[v + 1];
  if (e1 <= e0) return (V)0;
  const int64_t t0 = e0 / TL, t1 = (e1 - 1) / TL;
  V s = a.tail[t0];
  for (int64_t t = t0 + 1; t <= t1; ++t) s += a.head[t];
  return s;
}

template <typename V>
__device__ __forceinline__ V row_total(const TileArgs<V>& a, int64_t v) {
  return (a.span[v >> 5] >> (v & 31)) & 1u ? row_total_span(a, v) : a.s[v];
}

// the span bitmap: bit v set when row v is empty or its entries fall in
// more than one tile
__global__ void k_span_bits(int32_t n, const int64_t* __restrict__ rowptr, uint32_t* __restrict__ span,
                            uint32_t* __restrict__ nempty) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  bool f = false, e = false;
  if (v < n) {
    const int64_t e0 = rowptr[v], e1 = rowptr[v + 1];
    e = e1 <= e0;
    f = e || e0 / TL != (e1 - 1) / TL;
  }
  const uint32_t bits = __ballot_sync(0xffffffffu, f);
  const uint32_t empties = __ballot_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0 && v < n) {
    span[v >> 5] = bits;
    if (empties) atomicAdd(nempty, (uint32_t)__popc(empties));
  }
}

// FP64 s = W x by tiles (the residual of the refinement loop)
__global__ void __launch_bounds__(SV_T) k_tile_rowsum64(TileArgs<double> a, const double* __restrict__ x,
                                                        int64_t ntiles) {
  __shared__ TileSmem sm;
  tile_loop(a, x, ntiles, (int64_t)blockIdx.x * TL_W + (threadIdx.x >> 5), (int64_t)gridDim.x * TL_W,
            sm.off[threadIdx.x >> 5]);
}

// r = b - (sigma + alpha d_w) x + alpha s (r = b when x is zero); partial sums
// of r.r and b.b
__global__ void __launch_bounds__(SV_T) k_resid_rows(int32_t n, TileArgs<double> a, const double* __restrict__ dw,
                                                     double sigma, double alpha, const double* __restrict__ b,
                                                     const double* __restrict__ x, double* __restrict__ r,
                                                     double* __restrict__ prr, double* __restrict__ pbb, bool zero) {
  double rr = 0.0, bb = 0.0;
  for (int64_t v = (int64_t)blockIdx.x * SV_T + threadIdx.x; v < n; v += (int64_t)gridDim.x * SV_T) {
    const double ax = zero ? 0.0 : x[v] * (sigma + alpha * dw[v]) - alpha * row_total(a, v);
    const double rv = b[v] - ax;
    r[v] = rv;
    rr += rv * rv;
    bb += b[v] * b[v];
  }
  block_sum2(rr, bb);
  if (threadIdx.x == 0) {
    prr[blockIdx.x] = rr;
    pbb[blockIdx.x] = bb;
  }
}

// The whole inner CG in one cooperative launch (one launch per refinement
// step instead of nine per iteration).  An iteration:
//   A  s = W p by tiles                                        | grid barrier
//   B1 q = diag p - alpha s; partials of p.q                   | barrier
//   B2 d += a p, r -= a q, z = r prec; partials of r.z, r.r    | barrier
//   C  p = z + b p                                             | barrier
// Every block sums the partials itself in the same fixed order, so all
// blocks see the same scalars and leave the loop together (the inner
// tolerance rr <= tol2 rr0 is tested every iteration).  FP32 vectors, FP32
// per-thread partials, FP64 sums, as in the per-launch kernels.  The vectors
// start on 16-byte boundaries (B2 and C move four entries per access).
struct CG1 {
  int32_t n;
  int64_t ntiles;
  TileArgs<float> ta;
  const float* diag32;
  const float* prec;  // reciprocal diagonal (Jacobi) or null
  float alpha;
  Inner in;           // r, p, d from k_inner_init; q scratch
  double* part;       // [3][gridDim.x] block partials
  double rz0, rr0, tol2;
  int max_it;
  int* iters_out;
};

// sums of a[0..cnt) and b[0..cnt) in a fixed order (lane-strided, then a
// butterfly in warp 0), valid in every thread of the block; slot[2] is this
// call's own shared scratch (not reused before the next grid barrier)
__device__ __forceinline__ void block_fixed_sum2(const double* a, const double* b, int cnt, double* slot,
                                                 double& sa, double& sb) {
  if (threadIdx.x < 32) {
    double x = 0.0, y = 0.0;
#pragma unroll 4
    for (int i = threadIdx.x; i < cnt; i += 32) {
      x += a[i];
      if (b) y += b[i];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      x += __shfl_xor_sync(0xffffffffu, x, o);
      y += __shfl_xor_sync(0xffffffffu, y, o);
    }
    if (threadIdx.x == 0) {
      slot[0] = x;
      slot[1] = y;
    }
  }
  __syncthreads();
  sa = slot[0];
  sb = slot[1];
}

// FOLD (graphs without empty rows): phase A also finishes q and the p.q
// partials, and B1 disappears (three grid barriers per iteration); measured on
// GB300 with 80 registers (3 CTAs per SM; 64 spill): BA 2^20 4.35 -> 4.09 ms
// per solve, 2048^2 grid unchanged (10.7 ms: the tile phase takes longer by
// the per-row loads of p and the diagonal that B1 did in bulk)
template <bool FOLD>
__global__ void __launch_bounds__(SV_T, FOLD ? 3 : 4) k_cg1(CG1 c) {
  cgr::grid_group grid = cgr::this_grid();
  __shared__ TileSmem sm;
  __shared__ double slots[4];
  const int wid = threadIdx.x >> 5;
  const int G = gridDim.x;
  const int64_t gtid = (int64_t)blockIdx.x * SV_T + threadIdx.x;
  const int64_t gstride = (int64_t)G * SV_T;
  const int32_t n = c.n;
  const int64_t n4 = n / 4;
  float4* r4 = reinterpret_cast<float4*>(c.in.r);
  float4* p4 = reinterpret_cast<float4*>(c.in.p);
  float4* d4 = reinterpret_cast<float4*>(c.in.d);
  const float4* q4 = reinterpret_cast<const float4*>(c.in.q);
  const float4* m4 = reinterpret_cast<const float4*>(c.prec);
  const float4* g4 = reinterpret_cast<const float4*>(c.diag32);
  const float4* s4 = reinterpret_cast<const float4*>(c.ta.s);
  float4* q4w = reinterpret_cast<float4*>(c.in.q);
  double rz = c.rz0;
  int it = 0;
  const Fold fo{c.diag32, c.alpha, c.in.q};
  while (it < c.max_it) {
    float pqf = 0.0f;
    if (FOLD) {
      // A: q = diag p - alpha W p for the rows inside a tile, p.q partials
      tile_loop<float, true>(c.ta, c.in.p, c.ntiles, (int64_t)blockIdx.x * TL_W + wid, (int64_t)G * TL_W,
                             sm.off[wid], fo, &pqf);
    } else {
    // A: s = W p
    tile_loop(c.ta, c.in.p, c.ntiles, (int64_t)blockIdx.x * TL_W + wid, (int64_t)G * TL_W, sm.off[wid]);
    grid.sync();
    // B1: q = diag p - alpha s (rows marked in the span bitmap from their
    // tile partials)
    for (int64_t i = gtid; i < n4; i += gstride) {
      const float4 p = p4[i], dg = g4[i];
      float4 sv = s4[i];
      const uint32_t mk = (c.ta.span[i >> 3] >> ((i & 7) * 4)) & 0xFu;
      if (mk) {
        if (mk & 1u) sv.x = row_total_span(c.ta, 4 * i);
        if (mk & 2u) sv.y = row_total_span(c.ta, 4 * i + 1);
        if (mk & 4u) sv.z = row_total_span(c.ta, 4 * i + 2);
        if (mk & 8u) sv.w = row_total_span(c.ta, 4 * i + 3);
      }
      float4 q;
      q.x = p.x * dg.x - c.alpha * sv.x; q.y = p.y * dg.y - c.alpha * sv.y;
      q.z = p.z * dg.z - c.alpha * sv.z; q.w = p.w * dg.w - c.alpha * sv.w;
      q4w[i] = q;
      pqf = fmaf(p.x, q.x, pqf); pqf = fmaf(p.y, q.y, pqf);
      pqf = fmaf(p.z, q.z, pqf); pqf = fmaf(p.w, q.w, pqf);
    }
    for (int64_t v = 4 * n4 + gtid; v < n; v += gstride) {
      const float pv = c.in.p[v];
      const float qv = pv * c.diag32[v] - c.alpha * row_total(c.ta, v);
      c.in.q[v] = qv;
      pqf = fmaf(pv, qv, pqf);
    }
    }
    double pq = pqf, unused = 0.0;
    block_sum2(pq, unused);
    if (threadIdx.x == 0) c.part[blockIdx.x] = pq;
    grid.sync();
    double pq_t, unused2;
    block_fixed_sum2(c.part, nullptr, G, slots, pq_t, unused2);
    const float a = pq_t != 0.0 ? (float)(rz / pq_t) : 0.0f;
    // B2: d += a p, r -= a q
    float rzf = 0.0f, rrf = 0.0f;
    for (int64_t i = gtid; i < n4; i += gstride) {
      const float4 p = p4[i];
      float4 q = q4[i];
      float4 r = r4[i], d = d4[i];
      if (FOLD) {  // rows that cross tiles: q from their tile partials
        const uint32_t mk = (c.ta.span[i >> 3] >> ((i & 7) * 4)) & 0xFu;
        if (mk) {
          const float4 dg = g4[i];
          if (mk & 1u) q.x = p.x * dg.x - c.alpha * row_total_span(c.ta, 4 * i);
          if (mk & 2u) q.y = p.y * dg.y - c.alpha * row_total_span(c.ta, 4 * i + 1);
          if (mk & 4u) q.z = p.z * dg.z - c.alpha * row_total_span(c.ta, 4 * i + 2);
          if (mk & 8u) q.w = p.w * dg.w - c.alpha * row_total_span(c.ta, 4 * i + 3);
        }
      }
      d.x += a * p.x; d.y += a * p.y; d.z += a * p.z; d.w += a * p.w;
      r.x -= a * q.x; r.y -= a * q.y; r.z -= a * q.z; r.w -= a * q.w;
      d4[i] = d;
      r4[i] = r;
      const float4 m = c.prec ? m4[i] : make_float4(1.0f, 1.0f, 1.0f, 1.0f);
      rzf = fmaf(r.x, r.x * m.x, rzf); rzf = fmaf(r.y, r.y * m.y, rzf);
      rzf = fmaf(r.z, r.z * m.z, rzf); rzf = fmaf(r.w, r.w * m.w, rzf);
      rrf = fmaf(r.x, r.x, rrf); rrf = fmaf(r.y, r.y, rrf);
      rrf = fmaf(r.z, r.z, rrf); rrf = fmaf(r.w, r.w, rrf);
    }
    for (int64_t v = 4 * n4 + gtid; v < n; v += gstride) {
      c.in.d[v] += a * c.in.p[v];
      const float qv = FOLD && ((c.ta.span[v >> 5] >> (v & 31)) & 1u)
                           ? c.in.p[v] * c.diag32[v] - c.alpha * row_total_span(c.ta, v)
                           : c.in.q[v];
      const float rv = c.in.r[v] - a * qv;
      c.in.r[v] = rv;
      rzf = fmaf(rv, c.prec ? rv * c.prec[v] : rv, rzf);
      rrf = fmaf(rv, rv, rrf);
    }
    double rzn = rzf, rr = rrf;
    block_sum2(rzn, rr);
    if (threadIdx.x == 0) {
      c.part[G + blockIdx.x] = rzn;
      c.part[2 * G + blockIdx.x] = rr;
    }
    grid.sync();
    double rz_t, rr_t;
    block_fixed_sum2(c.part + G, c.part + 2 * G, G, slots + 2, rz_t, rr_t);
    ++it;
    if (rr_t <= c.tol2 * c.rr0) break;  // the same decision in every block
    // C: p = z + b p
    const float b = rz != 0.0 ? (float)(rz_t / rz) : 0.0f;
    for (int64_t i = gtid; i < n4; i += gstride) {
      const float4 r = r4[i];
      const float4 m = c.prec ? m4[i] : make_float4(1.0f, 1.0f, 1.0f, 1.0f);
      float4 p = p4[i];
      p.x = r.x * m.x + b * p.x; p.y = r.y * m.y + b * p.y;
      p.z = r.z * m.z + b * p.z; p.w = r.w * m.w + b * p.w;
      p4[i] = p;
    }
    for (int64_t v = 4 * n4 + gtid; v < n; v += gstride) {
      const float z = c.prec ? c.in.r[v] * c.prec[v] : c.in.r[v];
      c.in.p[v] = z + b * c.in.p[v];
    }
    rz = rz_t;
    grid.sync();
  }
  if (gtid == 0) *c.iters_out = it;
}

// ---------------------------------------------------------------------------
// Several right-hand sides (m >= 2): the solver's vectors interleaved by
// column, element (v, j) at v m + j.  A warp takes 32 VW columns of one row
// (VW values per lane), so each neighbour gather of the products loads one
// contiguous segment of 128 VW bytes (FP32).  Blocks are 32 x 8 threads (column
// x row), blockIdx.y is the column group; with fewer than 32 columns the block
// is LW x 256 / LW threads (LW the power of two from m on), several rows per
// warp.  Per-column partial sums go to part[j nb + blockIdx.x].
//
// The products run over row segments of at most IL_SEG entries: a warp that
// walked a whole hub row (11,600 entries at n = 2^19) held up the launch for
// about a millisecond.  A row of one segment is finished by its warp; the
// segments of a longer row leave partial sums that k_il_long_* adds in row
// order.  Bound by the neighbour gathers (DRAM and L2) and 8 vector passes per
// iteration.  Measured on GB300 (whole solves to 1e-12; before: a warp per row,
// one value per lane, 9 launches per iteration, and eight lanes per row below
// 32 columns): BA 2^19, 64 columns 75.4 -> 28.3 ms, 16 33.2 -> 10.8, 2 8.0 -> 3.6;
// weighted grid 2^20, 64 columns 132 -> 94; weighted R-MAT 2^16, 85 columns 76.7 ->
// 27; group closeness of n = 4099 (4096 columns) 28.4 -> 20.6.
// ---------------------------------------------------------------------------
constexpr int IL_T = 256;  // threads per block
constexpr int IL_SEG = 128;      // entries per segment, a warp per row (n = 5000, 21 columns: 2.7 ms, 3.2 with 256)
constexpr int IL_SEG_PACK = 64;  // and with several rows per warp (their segments run on few lanes)
constexpr int IL_U = 8;  // gathers of a warp in flight

template <typename T, int VW>
struct ILVec;
template <> struct ILVec<float, 1> { typedef float type; };
template <> struct ILVec<float, 2> { typedef float2 type; };
template <> struct ILVec<float, 4> { typedef float4 type; };
template <> struct ILVec<double, 1> { typedef double type; };
template <> struct ILVec<double, 2> { typedef double2 type; };

// VW consecutive columns of one row (aligned: VW divides m)
template <typename T, int VW>
__device__ __forceinline__ void il_load(const T* p, T (&x)[VW]) {
  const auto v = *reinterpret_cast<const typename ILVec<T, VW>::type*>(p);
  const T* s = reinterpret_cast<const T*>(&v);
#pragma unroll
  for (int c = 0; c < VW; ++c) x[c] = s[c];
}
template <typename T, int VW>
__device__ __forceinline__ void il_store(T* p, const T (&x)[VW]) {
  typename ILVec<T, VW>::type v;
  T* s = reinterpret_cast<T*>(&v);
#pragma unroll
  for (int c = 0; c < VW; ++c) s[c] = x[c];
  *reinterpret_cast<typename ILVec<T, VW>::type*>(p) = v;
}
// the same, leaving L2 first: vectors that are only streamed, so that the
// gathered one stays
template <typename T, int VW>
__device__ __forceinline__ void il_load_s(const T* p, T (&x)[VW]) {
  const auto v = __ldcs(reinterpret_cast<const typename ILVec<T, VW>::type*>(p));
  const T* s = reinterpret_cast<const T*>(&v);
#pragma unroll
  for (int c = 0; c < VW; ++c) x[c] = s[c];
}
template <typename T, int VW>
__device__ __forceinline__ void il_store_s(T* p, const T (&x)[VW]) {
  typename ILVec<T, VW>::type v;
  T* s = reinterpret_cast<T*>(&v);
#pragma unroll
  for (int c = 0; c < VW; ++c) s[c] = x[c];
  __stcs(reinterpret_cast<typename ILVec<T, VW>::type*>(p), v);
}

// per-column sums over the block's rows to pa (and pb), fixed order
template <int VW>
__device__ __forceinline__ void il_sum2(const double (&a)[VW], const double (&b)[VW], int j0, bool on,
                                        double* __restrict__ pa, double* __restrict__ pb, int nb, int blk) {
  constexpr int N = IL_T * VW + 128;  // rows of LW VW + 1 values, at most 128 rows
  __shared__ double sa[N], sb[N];
  const int ld = blockDim.x * VW + 1;
#pragma unroll
  for (int c = 0; c < VW; ++c) {
    sa[threadIdx.y * ld + threadIdx.x * VW + c] = a[c];
    sb[threadIdx.y * ld + threadIdx.x * VW + c] = b[c];
  }
  __syncthreads();
  for (int h = blockDim.y / 2; h > 0; h >>= 1) {
    if (threadIdx.y < h) {
#pragma unroll
      for (int c = 0; c < VW; ++c) {
        const int i = threadIdx.y * ld + threadIdx.x * VW + c;
        sa[i] += sa[i + h * ld];
        sb[i] += sb[i + h * ld];
      }
    }
    __syncthreads();
  }
  if (threadIdx.y == 0 && on) {
#pragma unroll
    for (int c = 0; c < VW; ++c) {
      pa[(size_t)(j0 + c) * nb + blk] = sa[threadIdx.x * VW + c];
      if (pb) pb[(size_t)(j0 + c) * nb + blk] = sb[threadIdx.x * VW + c];
    }
  }
}

// segments per row (at least one), and for rows of several their count and 1
__global__ void k_il_seg_count(int32_t n, int len, const int64_t* __restrict__ rowptr, uint32_t* __restrict__ cnt,
                               uint32_t* __restrict__ lcnt, uint32_t* __restrict__ lrow) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v > n) return;
  uint32_t c = 0;
  if (v < n) {
    const int64_t d = rowptr[v + 1] - rowptr[v];
    c = d > len ? (uint32_t)((d + len - 1) / len) : 1u;
  }
  cnt[v] = c;
  lcnt[v] = c > 1u ? c : 0u;
  lrow[v] = c > 1u ? 1u : 0u;
}

// segs: {row, entries, first entry, slot of its partial sum or -1}; longs:
// {row, first slot, slots, 0}; off: the exclusive scan of cnt, lcnt and lrow one
// after another (n + 1 entries each, the last of each 0; one scan and one copy
// of the totals instead of three: n = 5000, 3 columns 1733 -> 1614 us); tot: segments, slots and rows of several segments
__global__ void k_il_seg_fill(int32_t n, int len, const int64_t* __restrict__ rowptr, const uint32_t* __restrict__ off,
                              int4* __restrict__ segs, int4* __restrict__ longs, uint32_t* __restrict__ tot) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  const int64_t e0 = rowptr[v], e1 = rowptr[v + 1];
  const uint32_t *loff = off + n + 1, *lidx = loff + n + 1;
  const uint32_t o = off[v], c = off[v + 1] - o, l0 = loff[0], i0 = lidx[0];
  if (v == n - 1) {
    tot[0] = off[n];
    tot[1] = loff[n] - l0;
    tot[2] = lidx[n] - i0;
  }
  for (uint32_t k = 0; k < c; ++k) {
    const int64_t b = e0 + (int64_t)k * len;
    segs[o + k] = make_int4((int32_t)v, (int32_t)(e1 - b < len ? e1 - b : len), (int32_t)(uint32_t)b,
                            c > 1u ? (int32_t)(loff[v] - l0 + k) : -1);
  }
  if (c > 1u) longs[lidx[v] - i0] = make_int4((int32_t)v, (int32_t)(loff[v] - l0), (int32_t)c, 0);
}

// sum over a segment of w x[col] for VW columns, IL_U gathers in flight.  A
// full warp per row loads 32 column indices at a time and broadcasts them by
// shuffles; PACK (several rows per warp): every lane loads the index itself
// (one transaction per row).
template <typename T, int VW, bool PACK>
__device__ __forceinline__ void il_seg_sum(const int4& s, const int32_t* __restrict__ colidx,
                                           const float* __restrict__ w, const T* __restrict__ x, int m, int j0, bool on,
                                           T (&acc)[VW]) {
  const size_t e0 = (uint32_t)s.z;
#pragma unroll
  for (int c = 0; c < VW; ++c) acc[c] = (T)0;
  for (int b = 0; b < s.y; b += PACK ? IL_U : 32) {
    const int left = min(PACK ? IL_U : 32, s.y - b);
    int32_t cj = 0;
    T wj = (T)0;  // (converted before the broadcast: once per entry, not once per lane)
    if (!PACK && (int)threadIdx.x < left) {
      cj = __ldg(colidx + e0 + b + threadIdx.x);
      wj = w ? (T)__ldg(w + e0 + b + threadIdx.x) : (T)1;
    }
    for (int k = 0; k < left; k += IL_U) {
      T xv[IL_U][VW], ww[IL_U];
#pragma unroll
      for (int u = 0; u < IL_U; ++u) {
        int32_t c = 0;
        ww[u] = (T)0;
        if (PACK) {
          if (u < left) {
            c = __ldg(colidx + e0 + b + u);
            ww[u] = w ? (T)__ldg(w + e0 + b + u) : (T)1;
          }
        } else {
          c = __shfl_sync(0xffffffffu, cj, (k + u) & 31);
          ww[u] = __shfl_sync(0xffffffffu, wj, (k + u) & 31);
        }
        if (on && k + u < left) il_load<T, VW>(x + (size_t)c * m + j0, xv[u]);
        else {
#pragma unroll
          for (int q = 0; q < VW; ++q) xv[u][q] = (T)0;
        }
      }
#pragma unroll
      for (int u = 0; u < IL_U; ++u) {
        if (k + u < left) {
#pragma unroll
          for (int q = 0; q < VW; ++q) acc[q] += ww[u] * xv[u][q];
        }
      }
    }
  }
}

// dst[c ldd + i] = src[i lds + c] for i < rows, c < cols through 32 x 32 tiles:
// column-major [m][n] <-> interleaved [n][m].  *any (or null) = 1 where an entry
// differs from zero.
__global__ void k_il_transpose(int64_t rows, int64_t cols, const double* __restrict__ src, int64_t lds,
                               double* __restrict__ dst, int64_t ldd, uint32_t* __restrict__ any) {
  __shared__ double t[32][33];
  bool nz = false;
  for (int64_t br = blockIdx.y; br * 32 < rows; br += gridDim.y)
    for (int64_t bc = blockIdx.x; bc * 32 < cols; bc += gridDim.x) {
      for (int r = threadIdx.y; r < 32; r += blockDim.y) {
        const int64_t i = br * 32 + r, c = bc * 32 + threadIdx.x;
        if (i < rows && c < cols) {
          t[r][threadIdx.x] = src[i * lds + c];
          nz |= t[r][threadIdx.x] != 0.0;
        }
      }
      __syncthreads();
      for (int r = threadIdx.y; r < 32; r += blockDim.y) {
        const int64_t c = bc * 32 + r, i = br * 32 + threadIdx.x;
        if (i < rows && c < cols) dst[c * ldd + i] = t[threadIdx.x][r];
      }
      __syncthreads();
    }
  if (any && __syncthreads_or(nz) && threadIdx.x == 0 && threadIdx.y == 0) atomicOr(any, 1u);
}

// r = b - (sigma + alpha d_w) x + alpha s of one row
template <int VW>
__device__ __forceinline__ void il_resid_row(size_t i, double d, double alpha, const double (&acc)[VW],
                                             const double* __restrict__ b, const double* __restrict__ x,
                                             double* __restrict__ r, double (&rr)[VW], double (&bb)[VW]) {
  double bv[VW], xv[VW], rv[VW];
  il_load<double, VW>(b + i, bv);
  il_load<double, VW>(x + i, xv);
#pragma unroll
  for (int c = 0; c < VW; ++c) {
    rv[c] = bv[c] - (xv[c] * d - alpha * acc[c]);
    rr[c] += rv[c] * rv[c];
    bb[c] += bv[c] * bv[c];
  }
  il_store<double, VW>(r + i, rv);
}

template <int VW, bool PACK>
__global__ void __launch_bounds__(IL_T) k_il_resid(int m, int nseg, const int4* __restrict__ segs,
                                                  const int32_t* __restrict__ colidx, const float* __restrict__ w,
                                                  const double* __restrict__ dw, double sigma, double alpha,
                                                  const double* __restrict__ b, const double* __restrict__ x,
                                                  double* __restrict__ r, double* __restrict__ plong,
                                                  double* __restrict__ prr, double* __restrict__ pbb, int nb,
                                                  bool zero) {
  const int j0 = (int)(blockIdx.y * blockDim.x + threadIdx.x) * VW;
  const bool on = j0 < m;
  double rr[VW] = {}, bb[VW] = {};
  for (int g = blockIdx.x * blockDim.y + threadIdx.y; g < nseg; g += gridDim.x * blockDim.y) {
    int4 s = segs[g];
    if (zero) s.y = 0;  // x = 0: no products
    double acc[VW];
    il_seg_sum<double, VW, PACK>(s, colidx, w, x, m, j0, on, acc);
    if (!on) continue;
    if (s.w >= 0) il_store<double, VW>(plong + (size_t)s.w * m + j0, acc);
    else il_resid_row<VW>((size_t)s.x * m + j0, sigma + alpha * dw[s.x], alpha, acc, b, x, r, rr, bb);
  }
  il_sum2<VW>(rr, bb, j0, on, prr, pbb, nb, blockIdx.x);
}

// rows of several segments: their partial sums in row order
template <int VW>
__global__ void __launch_bounds__(IL_T) k_il_long_resid(int m, int nlong, const int4* __restrict__ longs,
                                                       const double* __restrict__ dw, double sigma, double alpha,
                                                       const double* __restrict__ b, const double* __restrict__ x,
                                                       double* __restrict__ r, const double* __restrict__ plong,
                                                       double* __restrict__ prr, double* __restrict__ pbb, int nb,
                                                       int blk0) {
  const int j0 = (int)(blockIdx.y * blockDim.x + threadIdx.x) * VW;
  const bool on = j0 < m;
  double rr[VW] = {}, bb[VW] = {};
  for (int g = blockIdx.x * blockDim.y + threadIdx.y; g < nlong && on; g += gridDim.x * blockDim.y) {
    const int4 s = longs[g];
    double acc[VW] = {};
    for (int k = 0; k < s.z; ++k) {
      double y[VW];
      il_load<double, VW>(plong + (size_t)(s.y + k) * m + j0, y);
#pragma unroll
      for (int c = 0; c < VW; ++c) acc[c] += y[c];
    }
    il_resid_row<VW>((size_t)s.x * m + j0, sigma + alpha * dw[s.x], alpha, acc, b, x, r, rr, bb);
  }
  il_sum2<VW>(rr, bb, j0, on, prr, pbb, nb, blk0 + blockIdx.x);
}

// r32 = r64 scale, p = z = r32 prec, d = 0; partials of r.z and r.r.  The
// element-wise kernels take IL_V rows per step.
constexpr int IL_V = 4;
template <int VW>
__global__ void __launch_bounds__(IL_T) k_il_init(int32_t n, int m, const double* __restrict__ r64,
                                                 const float* __restrict__ prec, const double* __restrict__ scal,
                                                 Inner in, double* __restrict__ prz, double* __restrict__ prr, int nb) {
  const int j0 = (int)(blockIdx.y * blockDim.x + threadIdx.x) * VW;
  const bool on = j0 < m;
  double sc[VW];
  float rz[VW] = {}, rr[VW] = {};  // per-thread partials in FP32, then FP64 across threads
#pragma unroll
  for (int c = 0; c < VW; ++c) sc[c] = on ? scal[(j0 + c) * 8 + 4] : 0.0;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.y + threadIdx.y; v < n && on; v += (int64_t)gridDim.x * blockDim.y) {
    const size_t i = (size_t)v * m + j0;
    const float pr = prec ? prec[v] : 1.0f;
    float r[VW], z[VW], zero[VW] = {};
#pragma unroll
    for (int c = 0; c < VW; ++c) {
      r[c] = (float)(r64[i + c] * sc[c]);
      z[c] = r[c] * pr;
      rz[c] = fmaf(r[c], z[c], rz[c]);
      rr[c] = fmaf(r[c], r[c], rr[c]);
    }
    il_store<float, VW>(in.r + i, r);
    il_store<float, VW>(in.p + i, z);
    il_store<float, VW>(in.d + i, zero);
  }
  double a[VW], b[VW];
#pragma unroll
  for (int c = 0; c < VW; ++c) {
    a[c] = rz[c];
    b[c] = rr[c];
  }
  il_sum2<VW>(a, b, j0, on, prz, prr, nb, blockIdx.x);
}

// q = diag p - alpha s of one row, partial of p.q
template <int VW>
__device__ __forceinline__ void il_spmv_row(size_t i, float dg, float alpha, const float (&acc)[VW], const Inner& in,
                                            float (&pq)[VW]) {
  float pv[VW], qv[VW];
  il_load<float, VW>(in.p + i, pv);
#pragma unroll
  for (int c = 0; c < VW; ++c) {
    qv[c] = pv[c] * dg - alpha * acc[c];
    pq[c] = fmaf(pv[c], qv[c], pq[c]);
  }
  il_store_s<float, VW>(in.q + i, qv);
}

// q = A p, partials of p.q
template <int VW, bool PACK>
__global__ void __launch_bounds__(IL_T) k_il_spmv(int m, int nseg, const int4* __restrict__ segs,
                                                 const int32_t* __restrict__ colidx, const float* __restrict__ w,
                                                 const float* __restrict__ diag32, float alpha, Inner in,
                                                 float* __restrict__ plong, double* __restrict__ ppq, int nb) {
  const int j0 = (int)(blockIdx.y * blockDim.x + threadIdx.x) * VW;
  const bool on = j0 < m;
  float pq[VW] = {};
  for (int g = blockIdx.x * blockDim.y + threadIdx.y; g < nseg; g += gridDim.x * blockDim.y) {
    const int4 s = segs[g];
    float acc[VW];
    il_seg_sum<float, VW, PACK>(s, colidx, w, in.p, m, j0, on, acc);
    if (!on) continue;
    if (s.w >= 0) il_store<float, VW>(plong + (size_t)s.w * m + j0, acc);
    else il_spmv_row<VW>((size_t)s.x * m + j0, diag32[s.x], alpha, acc, in, pq);
  }
  double a[VW], z[VW] = {};
#pragma unroll
  for (int c = 0; c < VW; ++c) a[c] = pq[c];
  il_sum2<VW>(a, z, j0, on, ppq, nullptr, nb, blockIdx.x);
}

template <int VW>
__global__ void __launch_bounds__(IL_T) k_il_long_spmv(int m, int nlong, const int4* __restrict__ longs,
                                                      const float* __restrict__ diag32, float alpha, Inner in,
                                                      const float* __restrict__ plong, double* __restrict__ ppq, int nb,
                                                      int blk0) {
  const int j0 = (int)(blockIdx.y * blockDim.x + threadIdx.x) * VW;
  const bool on = j0 < m;
  float pq[VW] = {};
  for (int g = blockIdx.x * blockDim.y + threadIdx.y; g < nlong && on; g += gridDim.x * blockDim.y) {
    const int4 s = longs[g];
    float acc[VW] = {};
    for (int k = 0; k < s.z; ++k) {
      float y[VW];
      il_load<float, VW>(plong + (size_t)(s.y + k) * m + j0, y);
#pragma unroll
      for (int c = 0; c < VW; ++c) acc[c] += y[c];
    }
    il_spmv_row<VW>((size_t)s.x * m + j0, diag32[s.x], alpha, acc, in, pq);
  }
  double a[VW], z[VW] = {};
#pragma unroll
  for (int c = 0; c < VW; ++c) a[c] = pq[c];
  il_sum2<VW>(a, z, j0, on, ppq, nullptr, nb, blk0 + blockIdx.x);
}

// r -= a q; partials of r.z and r.r (d += a p is left to k_il_p, which reads p
// anyway: 8 vector passes per iteration instead of 9)
template <int VW>
__global__ void __launch_bounds__(IL_T) k_il_update(int32_t n, int m, const float* __restrict__ prec,
                                                   const double* __restrict__ scal, Inner in, double* __restrict__ prz,
                                                   double* __restrict__ prr, int nb) {
  const int j0 = (int)(blockIdx.y * blockDim.x + threadIdx.x) * VW;
  const bool on = j0 < m;
  float a[VW], rz[VW] = {}, rr[VW] = {};
#pragma unroll
  for (int c = 0; c < VW; ++c) a[c] = on ? (float)scal[(j0 + c) * 8 + 6] : 0.0f;
  for (int64_t v0 = ((int64_t)blockIdx.x * blockDim.y + threadIdx.y) * IL_V; v0 < n && on;
       v0 += (int64_t)gridDim.x * blockDim.y * IL_V) {
    float r[IL_V][VW], q[IL_V][VW], pr[IL_V];
#pragma unroll
    for (int u = 0; u < IL_V; ++u) {
      if (v0 + u < n) {
        const size_t i = (size_t)(v0 + u) * m + j0;
        il_load_s<float, VW>(in.r + i, r[u]);
        il_load_s<float, VW>(in.q + i, q[u]);
        pr[u] = prec ? prec[v0 + u] : 1.0f;
      }
    }
#pragma unroll
    for (int u = 0; u < IL_V; ++u) {
      if (v0 + u < n) {
#pragma unroll
        for (int c = 0; c < VW; ++c) {
          r[u][c] -= a[c] * q[u][c];
          rz[c] = fmaf(r[u][c], r[u][c] * pr[u], rz[c]);
          rr[c] = fmaf(r[u][c], r[u][c], rr[c]);
        }
        il_store_s<float, VW>(in.r + (size_t)(v0 + u) * m + j0, r[u]);
      }
    }
  }
  double x[VW], y[VW];
#pragma unroll
  for (int c = 0; c < VW; ++c) {
    x[c] = rz[c];
    y[c] = rr[c];
  }
  il_sum2<VW>(x, y, j0, on, prz, prr, nb, blockIdx.x);
}

// d += a p; p = z + beta p
template <int VW>
__global__ void __launch_bounds__(IL_T) k_il_p(int32_t n, int m, const float* __restrict__ prec,
                                              const double* __restrict__ scal, Inner in) {
  const int j0 = (int)(blockIdx.y * blockDim.x + threadIdx.x) * VW;
  if (j0 >= m) return;
  float a[VW], beta[VW];
#pragma unroll
  for (int c = 0; c < VW; ++c) {
    a[c] = (float)scal[(j0 + c) * 8 + 6];
    beta[c] = (float)scal[(j0 + c) * 8 + 7];
  }
  for (int64_t v0 = ((int64_t)blockIdx.x * blockDim.y + threadIdx.y) * IL_V; v0 < n;
       v0 += (int64_t)gridDim.x * blockDim.y * IL_V) {
    float r[IL_V][VW], p[IL_V][VW], d[IL_V][VW], pr[IL_V];
#pragma unroll
    for (int u = 0; u < IL_V; ++u) {
      if (v0 + u < n) {
        const size_t i = (size_t)(v0 + u) * m + j0;
        il_load_s<float, VW>(in.r + i, r[u]);
        il_load<float, VW>(in.p + i, p[u]);
        il_load_s<float, VW>(in.d + i, d[u]);
        pr[u] = prec ? prec[v0 + u] : 1.0f;
      }
    }
#pragma unroll
    for (int u = 0; u < IL_V; ++u) {
      if (v0 + u < n) {
        const size_t i = (size_t)(v0 + u) * m + j0;
#pragma unroll
        for (int c = 0; c < VW; ++c) {
          d[u][c] += a[c] * p[u][c];
          p[u][c] = r[u][c] * pr[u] + beta[c] * p[u][c];
        }
        il_store_s<float, VW>(in.d + i, d[u]);
        il_store<float, VW>(in.p + i, p[u]);
      }
    }
  }
}

// x += d / scale (FP64), only for active columns
template <int VW>
__global__ void __launch_bounds__(IL_T) k_il_correct(int32_t n, int m, const double* __restrict__ scal,
                                                    const float* __restrict__ d, double* __restrict__ x) {
  const int j0 = (int)(blockIdx.y * blockDim.x + threadIdx.x) * VW;
  if (j0 >= m) return;
  double f[VW];  // one division per thread: GB300's FP64 rate is low
#pragma unroll
  for (int c = 0; c < VW; ++c) f[c] = scal[(j0 + c) * 8 + 5] != 0.0 ? 1.0 / scal[(j0 + c) * 8 + 4] : 0.0;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.y + threadIdx.y; v < n; v += (int64_t)gridDim.x * blockDim.y) {
    const size_t i = (size_t)v * m + j0;
    float dv[VW];
    il_load<float, VW>(d + i, dv);
#pragma unroll
    for (int c = 0; c < VW; ++c)
      if (f[c] != 0.0) x[i + c] += (double)dv[c] * f[c];
  }
}

// sum of part[0..nb) by one warp, fixed order, valid in every lane
__device__ __forceinline__ double il_warp_sum(const double* __restrict__ part, int nb) {
  double s[4] = {};
  for (int i = threadIdx.x & 31; i < nb; i += 128) {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (i + 32 * k < nb) s[k] += part[i + 32 * k];
  }
  double x = (s[0] + s[2]) + (s[1] + s[3]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// Per-column scalars after the products: pq and a = rz / pq (a warp per column;
// a block per column took 19 us for 4096 columns; 2176 take 8 now).
constexpr int IL_SW = 4;  // warps per block
__global__ void __launch_bounds__(32 * IL_SW) k_il_alpha(int m, const double* __restrict__ ppq, int nb,
                                                        double* __restrict__ scal) {
  const int j = blockIdx.x * IL_SW + (threadIdx.x >> 5);
  if (j >= m) return;
  const double pq = il_warp_sum(ppq + (size_t)j * nb, nb);
  if ((threadIdx.x & 31) == 0) {
    double* sc = scal + (size_t)j * 8;
    sc[1] = pq;
    sc[6] = (sc[5] != 0.0 && pq != 0.0) ? sc[0] / pq : 0.0;
  }
}

// After the update: the new r.z and r.r, beta = rz_new / rz, rz <- rz_new.
__global__ void __launch_bounds__(32 * IL_SW) k_il_beta(int m, const double* __restrict__ prz,
                                                       const double* __restrict__ prr, int nb,
                                                       double* __restrict__ scal, double* __restrict__ rr_out) {
  const int j = blockIdx.x * IL_SW + (threadIdx.x >> 5);
  if (j >= m) return;
  const double rz = il_warp_sum(prz + (size_t)j * nb, nb);
  const double rr = il_warp_sum(prr + (size_t)j * nb, nb);
  if ((threadIdx.x & 31) == 0) {
    double* sc = scal + (size_t)j * 8;
    sc[7] = sc[0] != 0.0 ? rz / sc[0] : 0.0;
    sc[0] = rz;
    sc[2] = rz;
    sc[3] = rr;
    rr_out[j] = rr;
  }
}

// The interleaved kernels for VW columns per lane, and the plan of a solve.
struct ILPlan {
  int vw, lw;            // columns per lane, lanes per row
  int gy, gxs, gxl, gxe;  // column groups, blocks over segments, long rows and rows
  int nseg, nlong, nslot;
  const int4* segs;
  const int4* longs;
  void* plong;                // [nslot][m] partial sums (FP64 or FP32)
};

template <int VW>
static void il_launch_resid(const ILPlan& pl, const fc_graph* g, int m, double sigma, double alpha, const double* b,
                            const double* x, double* r, double* pA, double* pB, bool zero, cudaStream_t st) {
  const dim3 blk(pl.lw, IL_T / pl.lw);
  const int nb = pl.gxs + pl.gxl;
  auto* kern = pl.lw == 32 ? k_il_resid<VW, false> : k_il_resid<VW, true>;
  kern<<<dim3(pl.gxs, pl.gy), blk, 0, st>>>(m, pl.nseg, pl.segs, g->colidx, g->w, g->dw, sigma, alpha, b, x, r,
                                            (double*)pl.plong, pA, pB, nb, zero);
  note_launch();
  if (pl.nlong > 0) {
    k_il_long_resid<VW><<<dim3(pl.gxl, pl.gy), blk, 0, st>>>(m, pl.nlong, pl.longs, g->dw, sigma, alpha, b, x, r,
                                                             (const double*)pl.plong, pA, pB, nb, pl.gxs);
    note_launch();
  }
}

template <int VW>
static void il_launch_init(const ILPlan& pl, int32_t n, int m, const double* r64, const float* prec,
                           const double* scal, const Inner& in, double* pA, double* pB, cudaStream_t st) {
  k_il_init<VW><<<dim3(pl.gxe, pl.gy), dim3(pl.lw, IL_T / pl.lw), 0, st>>>(n, m, r64, prec, scal, in, pA, pB, pl.gxe);
  note_launch();
}

// one inner iteration
template <int VW>
static void il_launch_iter(const ILPlan& pl, const fc_graph* g, int m, const float* prec, const float* diag32,
                           float alpha, double* scal, const Inner& in, double* pA, double* pB, double* rr_out,
                           cudaStream_t st) {
  const dim3 blk(pl.lw, IL_T / pl.lw);
  const int nb = pl.gxs + pl.gxl;
  auto* kern = pl.lw == 32 ? k_il_spmv<VW, false> : k_il_spmv<VW, true>;
  kern<<<dim3(pl.gxs, pl.gy), blk, 0, st>>>(m, pl.nseg, pl.segs, g->colidx, g->w, diag32, alpha, in, (float*)pl.plong,
                                            pA, nb);
  if (pl.nlong > 0) {
    k_il_long_spmv<VW><<<dim3(pl.gxl, pl.gy), blk, 0, st>>>(m, pl.nlong, pl.longs, diag32, alpha, in,
                                                            (const float*)pl.plong, pA, nb, pl.gxs);
    note_launch();
  }
  k_il_alpha<<<(m + IL_SW - 1) / IL_SW, 32 * IL_SW, 0, st>>>(m, pA, nb, scal);
  k_il_update<VW><<<dim3(pl.gxe, pl.gy), blk, 0, st>>>(g->n, m, prec, scal, in, pA, pB, pl.gxe);
  k_il_beta<<<(m + IL_SW - 1) / IL_SW, 32 * IL_SW, 0, st>>>(m, pA, pB, pl.gxe, scal, rr_out);
  k_il_p<VW><<<dim3(pl.gxe, pl.gy), blk, 0, st>>>(g->n, m, prec, scal, in);
  for (int i = 0; i < 5; ++i) note_launch();
}

template <int VW>
static void il_launch_correct(const ILPlan& pl, int32_t n, int m, const double* scal, const float* d, double* x,
                              cudaStream_t st) {
  k_il_correct<VW><<<dim3(pl.gxe, pl.gy), dim3(pl.lw, IL_T / pl.lw), 0, st>>>(n, m, scal, d, x);
  note_launch();
}

// Columns of a solve with n_rhs right-hand sides.  Values per lane: a warp takes
// up to 64 columns, and 128 in 16-byte accesses from 128 on.  The columns are
// filled up with zero columns (never active) to a multiple of them (R-MAT 2^16:
// 33 columns 12.9 ms, 63 17.6 -> 13.4 against one value per lane; 96 columns 19.7
// with two values, 21.6 with four; filling up to 8 or 16 columns changes less
// than 5% either way).
static int il_values(int n_rhs) { return n_rhs >= 128 ? 4 : n_rhs > 32 ? 2 : 1; }
static int il_columns(int n_rhs) {
  const int pad = il_values(n_rhs) - 1;
  return n_rhs + pad <= 65535 ? (n_rhs + pad) & ~pad : n_rhs;
}

// Bytes of the partial sums of rows of several segments of `len` entries, at
// most: only rows longer than len have them, fewer than 2 d / len each.
static size_t il_long_bytes(const fc_graph* g, int len, int m) {
  return g->max_deg <= len ? 0 : (size_t)(2 * g->nnz / len + 1) * m * sizeof(double);
}

// Entries per segment: IL_SEG or IL_SEG_PACK, doubled while the partial sums
// could take more than an FP64 vector block and IL_LONG bytes.  Sparse graphs
// (mean degree up to len / 2) never are; on a complete graph of n = 20,000 the
// sums of 4096 columns would take 100 GB.
constexpr size_t IL_LONG = 256u << 20;
static int il_seg_len(const fc_graph* g, int m) {
  int len = m > 16 ? IL_SEG : IL_SEG_PACK;
  const size_t most = std::max(IL_LONG, (size_t)g->n * m * sizeof(double));
  while (il_long_bytes(g, len, m) > most) len *= 2;
  return len;
}

#define IL_DISPATCH(vw, call4, call2, call1) \
  do {                                       \
    if ((vw) == 4) call4;                    \
    else if ((vw) == 2) call2;               \
    else call1;                              \
  } while (0)

// FP64 residual and copies of b and x, four FP32 vectors, and what the rows need
size_t solve_scratch_bytes(const fc_graph* g, int32_t n_rhs) {
  const int m = il_columns(n_rhs), len = il_seg_len(g, m);
  const size_t n = (size_t)g->n, lmax = (size_t)(g->nnz / len) + 1;
  return n * m * 40 + il_long_bytes(g, len, m) + (n + 2 * lmax) * 16 + n * 32 + (16u << 20) + (size_t)m * 64;
}

}  // namespace fcx

using namespace fcx;

// Scratch of a call of several columns: 40 bytes per column and vertex.
static fc_status solve_columns(fc_graph* g, int32_t alpha_idx, const double* b, double* x, int32_t n_rhs,
                               double rel_tol, int32_t max_iter, int32_t* iters_out, cudaStream_t st, bool jacobi,
                               double sigma) {
  const int32_t n = g->n;
  const int vw = il_values(n_rhs), m = il_columns(n_rhs);
  const double alpha = g->alphas[alpha_idx];
  const int nb = (n + SV_T - 1) / SV_T;  // blocks of the element-wise kernels
  const size_t nm = (size_t)n * m;
  int coop = 0;
  FC_CK(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, g->device));
  // several right-hand sides: vectors interleaved by column; one: edge tiles
  // and the inner CG in one cooperative launch
  const bool il = m >= 2 || !coop;
  ILPlan il32{}, il64{};  // FP32 products and vectors, FP64 residual
  // scratch: FP64 r64, FP32 r/p/q/d, diag32, partials, scalars
  CallScratch scr(st);
  double* r64 = nullptr;
  float* f32 = nullptr;
  double* part = nullptr;
  double* scal = nullptr;
  // each FP32 vector starts on a 16-byte boundary (four-wide accesses)
  const size_t nmp = (nm + 3) & ~(size_t)3, np4 = ((size_t)n + 3) & ~(size_t)3;
  FC_CK(scr.get(&r64, nm * sizeof(double)));
  FC_CK(scr.get(&f32, (4 * nmp + 2 * np4) * sizeof(float)));
  // partial sums per column of the column-major kernels: a few thousand blocks in all
  const int nbx = std::max(1, std::min(nb, 2048 / m));
  int npart = nbx;
  double* bi = nullptr;  // interleaved copies of b and x
  double* xi = nullptr;
  void* seg_mem = nullptr;
  void* plong = nullptr;
  const int gy = (m + 31) / 32;  // column tiles of the transposes
  uint32_t h_any = 1;  // x differs from zero on entry
  if (il) {
    uint32_t* any = nullptr;  // [0] x differs from zero, [1..3] counts of the row segments
    FC_CK(scr.get(&any, 16));
    FC_CK(cudaMemsetAsync(any, 0, 16, st));
    FC_CK(scr.get(&bi, nm * sizeof(double)));
    FC_CK(scr.get(&xi, nm * sizeof(double)));
    if (m != n_rhs) {
      FC_CK(cudaMemsetAsync(bi, 0, nm * sizeof(double), st));
      FC_CK(cudaMemsetAsync(xi, 0, nm * sizeof(double), st));
    }
    const dim3 tg((unsigned)std::min<int64_t>((n + 31) / 32, 1024), (unsigned)std::min<int64_t>(gy, 1024));
    k_il_transpose<<<tg, dim3(32, 8), 0, st>>>(n_rhs, n, b, n, bi, m, nullptr);
    FC_LAUNCHED();
    k_il_transpose<<<tg, dim3(32, 8), 0, st>>>(n_rhs, n, x, n, xi, m, any);
    FC_LAUNCHED();
    // row segments (k_il_seg_count, _fill)
    const int len = il_seg_len(g, m);
    const size_t n1 = (size_t)n + 1, lmax = (size_t)(g->nnz / len) + 1, smax = (size_t)n + lmax;
    FC_CK(scr.get(&seg_mem, (smax + lmax) * 16 + n1 * 4 * 6));
    int4* segs = (int4*)seg_mem;
    int4* longs = segs + smax;
    uint32_t* cnt = (uint32_t*)(longs + lmax);
    uint32_t *lcnt = cnt + n1, *lrow = cnt + 2 * n1, *off = cnt + 3 * n1;
    k_il_seg_count<<<(unsigned)((n1 + 255) / 256), 256, 0, st>>>(n, len, g->rowptr, cnt, lcnt, lrow);
    FC_LAUNCHED();
    const fc_status ss = exclusive_scan(cnt, off, (int64_t)(3 * n1), st);
    if (ss != FC_OK) return ss;
    k_il_seg_fill<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, len, g->rowptr, off, segs, longs, any + 1);
    FC_LAUNCHED();
    uint32_t ha[4];
    FC_CK(cudaMemcpyAsync(ha, any, 16, cudaMemcpyDeviceToHost, st));
    FC_CK(cudaStreamSynchronize(st));
    h_any = ha[0];
    const uint32_t* h = ha + 1;
    FC_CK(scr.get(&plong, std::max<size_t>(1, (size_t)h[1] * m * sizeof(double))));
    int nsm = 0;
    FC_CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, g->device));
    auto plan = [&](int vw) {
      ILPlan p;
      p.vw = vw;
      // (two lanes per row leave small graphs with too few warps: n = 5000,
      // two columns 2.6 ms against 2.3 ms on four lanes; 2^19: 3.7 against 4.5)
      p.lw = n < (1 << 16) ? 4 : 2;
      while (p.lw < 32 && p.lw < m) p.lw *= 2;
      const int rows = IL_T / p.lw;
      p.gy = (m + p.lw * vw - 1) / (p.lw * vw);
      const int tot = std::max(1, nsm * 16 / p.gy);  // blocks per column group: about 16 per SM in all
      p.nseg = (int)h[0];
      p.nslot = (int)h[1];
      p.nlong = (int)h[2];
      p.gxs = std::max(1, std::min((p.nseg + rows - 1) / rows, tot));
      p.gxl = p.nlong > 0 ? std::max(1, std::min((p.nlong + rows - 1) / rows, tot)) : 0;
      p.gxe = std::max(1, std::min((n + rows * IL_V - 1) / (rows * IL_V), tot));
      p.segs = segs;
      p.longs = longs;
      p.plong = plong;
      npart = std::max(npart, std::max(p.gxs + p.gxl, p.gxe));
      return p;
    };
    il32 = plan(m % vw == 0 ? vw : 1);
    il64 = plan(m % vw == 0 ? std::min(vw, 2) : 1);
  }
  const double* bv = il ? bi : b;
  double* xv = il ? xi : x;
  FC_CK(scr.get(&part, (size_t)2 * m * npart * sizeof(double) + 4 * m * sizeof(double)));
  FC_CK(scr.get(&scal, (size_t)8 * m * sizeof(double)));
  Inner in;
  in.r = f32;
  in.p = f32 + nmp;
  in.q = f32 + 2 * nmp;
  in.d = f32 + 3 * nmp;
  in.scal = scal;
  float* diag32 = f32 + 4 * nmp;
  float* inv32 = diag32 + np4;  // the reciprocal of the diagonal
  double* pA = part;
  double* pB = part + (size_t)m * npart;
  double* sums = part + (size_t)2 * m * npart;  // [0..m): rr, [m..2m): bb
  const float* prec = jacobi ? inv32 : nullptr;  // z = r * prec
  k_diag32<<<(n + 255) / 256, 256, 0, st>>>(n, g->dw, sigma, alpha, diag32, inv32);
  FC_LAUNCHED();
  const double inner_tol = 1e-4;
  const int check_every = 8;
  // one right-hand side: row sums by edge tiles (FP64 residual and FP32
  // inner products) and the cooperative inner CG (every CTA resident)
  const bool tiles = !il;
  const int64_t ntiles = (g->nnz + TL - 1) / TL;
  TileArgs<double> t64{};
  TileArgs<float> t32{};
  void* tile_mem = nullptr;
  int tile_grid = 0;
  bool fold = false;  // q and p.q in the tile phase (graphs without empty rows)
  int cg1_grid = 0;
  double* cg1_part = nullptr;
  if (tiles) {
    const size_t nt = (size_t)std::max<int64_t>(ntiles, 1);
    // [s32 n4][s64 n4][head64 nt][tail64 nt][head32 nt][tail32 nt][row0 nt][row1 nt][meta nt TL_T][span]
    const size_t nsw = ((size_t)n + 31) / 32;
    const size_t bytes = np4 * 12 + nt * 16 + nt * 8 + nt * 8 + nt * TL_T * 4 + nsw * 4 + 16;
    FC_CK(scr.get(&tile_mem, bytes));
    t32.s = (float*)tile_mem;  // 16-byte aligned: B1 reads it four-wide
    t64.s = (double*)(t32.s + np4);
    t64.head = t64.s + np4;
    t64.tail = t64.head + nt;
    t32.head = (float*)(t64.tail + nt);
    t32.tail = t32.head + nt;
    int32_t* row0 = (int32_t*)(t32.tail + nt);
    int32_t* row1 = row0 + nt;
    uint32_t* meta = (uint32_t*)(row1 + nt);
    uint32_t* span = meta + nt * TL_T;
    uint32_t* nempty = span + nsw;  // rows without entries
    const bool vec = ((uintptr_t)g->colidx % 16 == 0) && (g->w == nullptr || (uintptr_t)g->w % 16 == 0);
    t64.nnz = g->nnz;
    t64.rowptr = g->rowptr;
    t64.colidx = g->colidx;
    t64.w = g->w;
    t64.row0 = row0;
    t64.row1 = row1;
    t64.meta = meta;
    t64.span = span;
    t64.vec = vec;
    t32.nnz = g->nnz;
    t32.rowptr = g->rowptr;
    t32.colidx = g->colidx;
    t32.w = g->w;
    t32.row0 = row0;
    t32.row1 = row1;
    t32.meta = meta;
    t32.span = span;
    t32.vec = vec;
    if (ntiles > 0) {
      k_tile_rows<<<(unsigned)((2 * ntiles + 255) / 256), 256, 0, st>>>(n, g->nnz, g->rowptr, ntiles, row0, row1);
      FC_LAUNCHED();
      k_tile_meta<<<(unsigned)std::min<int64_t>((ntiles + TL_W - 1) / TL_W, 4096), SV_T, 0, st>>>(
          g->nnz, g->rowptr, ntiles, row0, row1, meta);
      FC_LAUNCHED();
    }
    uint32_t* any = nempty + 1;      // x differs from zero on entry
    FC_CK(cudaMemsetAsync(nempty, 0, 2 * sizeof(uint32_t), st));
    k_span_bits<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, g->rowptr, span, nempty);
    FC_LAUNCHED();
    k_any_nonzero<<<(unsigned)std::min<int64_t>((n + 255) / 256, 152 * 8), 256, 0, st>>>(n, x, any);
    FC_LAUNCHED();
    uint32_t h2[2];
    FC_CK(cudaMemcpyAsync(h2, nempty, sizeof(h2), cudaMemcpyDeviceToHost, st));
    FC_CK(cudaStreamSynchronize(st));
    fold = h2[0] == 0;
    h_any = h2[1];
    int per_sm = 0, nsm = 0;
    FC_CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, g->device));
    tile_grid = (int)std::max<int64_t>(1, std::min<int64_t>((ntiles + TL_W - 1) / TL_W, (int64_t)8 * nsm));
    FC_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fold ? k_cg1<true> : k_cg1<false>, SV_T, 0));
    cg1_grid = std::max(1, std::min(per_sm, 8)) * nsm;
    FC_CK(scr.get(&cg1_part, (3 * (size_t)cg1_grid + 1) * sizeof(double)));
  }
  std::vector<double> h_rr(m), h_bb(m), h_scal((size_t)8 * m, 0.0), h_in(m);
  int used = 0;
  fc_status result = FC_ENOCONV;
  for (int outer = 0; outer < 64; ++outer) {
    const bool zero = outer == 0 && h_any == 0;  // x = 0: the residual is b
    const int nres = il ? il64.gxs + il64.gxl : nbx;  // residual partials per column
    if (il) {
      if (il64.vw == 2) il_launch_resid<2>(il64, g, m, sigma, alpha, bv, xv, r64, pA, pB, zero, st);
      else il_launch_resid<1>(il64, g, m, sigma, alpha, bv, xv, r64, pA, pB, zero, st);
    } else {
      if (ntiles > 0 && !zero) {
        k_tile_rowsum64<<<tile_grid, SV_T, 0, st>>>(t64, x, ntiles);
        FC_LAUNCHED();
      }
      k_resid_rows<<<nbx, SV_T, 0, st>>>(n, t64, g->dw, sigma, alpha, b, x, r64, pA, pB, zero);
    }
    FC_LAUNCHED();
    k_colsum<<<m, SV_T, 0, st>>>(pA, nres, sums);
    fcx::note_launch();
    k_colsum<<<m, SV_T, 0, st>>>(pB, nres, sums + m);
    fcx::note_launch();
    if (sigma == 0.0) {  // singular L: keep the residual in L's range
      const fc_status sc = center_columns(n, m, r64, il ? m : 1, il ? 1 : n, r64, sums, pA, nbx, st);
      if (sc != FC_OK) return sc;
    }
    FC_CK(cudaMemcpyAsync(h_rr.data(), sums, m * sizeof(double), cudaMemcpyDeviceToHost, st));
    FC_CK(cudaMemcpyAsync(h_bb.data(), sums + m, m * sizeof(double), cudaMemcpyDeviceToHost, st));
    FC_CK(cudaStreamSynchronize(st));
    bool all_ok = true;
    for (int j = 0; j < m; ++j) {
      const double rn = std::sqrt(h_rr[j]), bn = std::sqrt(h_bb[j]);
      const bool ok = rn <= rel_tol * bn || rn == 0.0;
      h_scal[(size_t)j * 8 + 5] = ok ? 0.0 : 1.0;
      h_scal[(size_t)j * 8 + 4] = rn > 0.0 ? 1.0 / rn : 1.0;
      all_ok = all_ok && ok;
    }
    if (all_ok) {
      result = FC_OK;
      break;
    }
    if (used >= max_iter) break;
    FC_CK(cudaMemcpyAsync(scal, h_scal.data(), (size_t)8 * m * sizeof(double), cudaMemcpyHostToDevice, st));
    if (il)
      IL_DISPATCH(il32.vw, il_launch_init<4>(il32, n, m, r64, prec, scal, in, pA, pB, st),
                  il_launch_init<2>(il32, n, m, r64, prec, scal, in, pA, pB, st),
                  il_launch_init<1>(il32, n, m, r64, prec, scal, in, pA, pB, st));
    else
      k_inner_init<<<nbx, SV_T, 0, st>>>(n, r64, prec, scal, in, pA, pB, nbx);
    FC_LAUNCHED();
    k_colsum<<<m, SV_T, 0, st>>>(pA, il ? il32.gxe : nbx, sums);
    fcx::note_launch();
    k_colsum<<<m, SV_T, 0, st>>>(pB, il ? il32.gxe : nbx, sums + m);
    fcx::note_launch();
    FC_CK(cudaMemcpyAsync(h_in.data(), sums, m * sizeof(double), cudaMemcpyDeviceToHost, st));
    FC_CK(cudaMemcpyAsync(h_rr.data(), sums + m, m * sizeof(double), cudaMemcpyDeviceToHost, st));
    FC_CK(cudaStreamSynchronize(st));
    std::vector<double> rr0(h_rr);
    for (int j = 0; j < m; ++j) h_scal[(size_t)j * 8 + 0] = h_in[j];
    FC_CK(cudaMemcpyAsync(scal, h_scal.data(), (size_t)8 * m * sizeof(double), cudaMemcpyHostToDevice, st));
    if (cg1_grid > 0) {
      // one right-hand side: the inner CG in one cooperative launch
      CG1 c;
      c.n = n;
      c.ntiles = ntiles;
      c.ta = t32;
      c.diag32 = diag32;
      c.prec = prec;
      c.alpha = (float)alpha;
      c.in = in;
      c.part = cg1_part;
      c.rz0 = h_in[0];
      c.rr0 = rr0[0];
      c.tol2 = inner_tol * inner_tol;
      c.max_it = max_iter - used;
      c.iters_out = (int*)(cg1_part + 3 * cg1_grid);
      void* args[] = {&c};
      FC_CK(cudaLaunchCooperativeKernel(fold ? (void*)k_cg1<true> : (void*)k_cg1<false>, dim3(cg1_grid),
                                        dim3(SV_T), args, 0, st));
      FC_LAUNCHED();
      int done = 0;
      FC_CK(cudaMemcpyAsync(&done, c.iters_out, sizeof(int), cudaMemcpyDeviceToHost, st));
      FC_CK(cudaStreamSynchronize(st));
      used += done;
    }
    int it = 0;
    while (il && used < max_iter) {
      IL_DISPATCH(il32.vw, il_launch_iter<4>(il32, g, m, prec, diag32, (float)alpha, scal, in, pA, pB, sums + m, st),
                  il_launch_iter<2>(il32, g, m, prec, diag32, (float)alpha, scal, in, pA, pB, sums + m, st),
                  il_launch_iter<1>(il32, g, m, prec, diag32, (float)alpha, scal, in, pA, pB, sums + m, st));
      FC_CK(cudaGetLastError());
      ++used;
      ++it;
      if (it == 1 || it == 2 || it == 4 || it % check_every == 0) {
        FC_CK(cudaMemcpyAsync(h_rr.data(), sums + m, m * sizeof(double), cudaMemcpyDeviceToHost, st));
        FC_CK(cudaStreamSynchronize(st));
        bool conv = true;
        for (int j = 0; j < m; ++j)
          if (h_scal[(size_t)j * 8 + 5] != 0.0 && std::sqrt(h_rr[j]) > inner_tol * std::sqrt(rr0[j])) conv = false;
        if (conv) break;
      }
    }
    if (il)
      IL_DISPATCH(il32.vw, il_launch_correct<4>(il32, n, m, scal, in.d, xv, st),
                  il_launch_correct<2>(il32, n, m, scal, in.d, xv, st),
                  il_launch_correct<1>(il32, n, m, scal, in.d, xv, st));
    else
      k_correct<<<nbx, SV_T, 0, st>>>(n, scal, in.d, x);
    FC_LAUNCHED();
  }
  if (il) {
    const dim3 tg((unsigned)std::min<int64_t>(gy, 1024), (unsigned)std::min<int64_t>((n + 31) / 32, 1024));
    k_il_transpose<<<tg, dim3(32, 8), 0, st>>>(n, n_rhs, xi, m, x, n, nullptr);
    FC_LAUNCHED();
  }
  scr.release();
  FC_CK(cudaStreamSynchronize(st));
  if (iters_out) *iters_out = used;
  if (result != FC_OK) set_error("fc_solve: max_iter reached before rel_tol");
  return result;
}

// The columns are independent: where the scratch of all of them does not fit
// (nothing has been written to x then), they are solved in halves.
static fc_status solve_impl(fc_graph* g, int32_t alpha_idx, const double* b, double* x, int32_t n_rhs,
                            double rel_tol, int32_t max_iter, int32_t* iters_out, cudaStream_t st, bool jacobi,
                            double sigma = 1.0) {
  if (g == nullptr || b == nullptr || x == nullptr || n_rhs < 1 || n_rhs > 65535 || alpha_idx < 0 ||
      alpha_idx >= g->n_alpha || !(rel_tol > 0.0) || max_iter < 1) {
    set_error("fc_solve: bad argument");
    return FC_EINVAL;
  }
  const fc_status s =
      solve_columns(g, alpha_idx, b, x, n_rhs, rel_tol, max_iter, iters_out, st, jacobi, sigma);
  if (s != FC_ENOMEM || n_rhs == 1) return s;
  const int32_t h = n_rhs / 2;
  int32_t it[2] = {0, 0};
  const size_t off = (size_t)h * g->n;
  const fc_status s0 = solve_impl(g, alpha_idx, b, x, h, rel_tol, max_iter, &it[0], st, jacobi, sigma);
  if (s0 != FC_OK && s0 != FC_ENOCONV) return s0;
  const fc_status s1 = solve_impl(g, alpha_idx, b + off, x + off, n_rhs - h, rel_tol, max_iter, &it[1], st, jacobi, sigma);
  if (iters_out) *iters_out = std::max(it[0], it[1]);
  return s1 != FC_OK ? s1 : s0;
}

extern "C" fc_status fc_solve(fc_graph* g, int32_t alpha_idx, const double* b, double* x, int32_t n_rhs,
                              double rel_tol, int32_t max_iter, int32_t* iters_out, void* stream) {
  return solve_impl(g, alpha_idx, b, x, n_rhs, rel_tol, max_iter, iters_out, (cudaStream_t)stream, true);
}

extern "C" fc_status fc_pivot_solve(fc_graph* g, int32_t alpha_idx, double* x, double rel_tol, int32_t max_iter,
                                    int32_t* iters_out, void* stream) {
  if (g == nullptr || x == nullptr || alpha_idx < 0 || alpha_idx >= g->n_alpha) {
    set_error("fc_pivot_solve: bad argument");
    return FC_EINVAL;
  }
  cudaStream_t st = (cudaStream_t)stream;
  const int32_t n = g->n;
  double* rhs = nullptr;
  double* part = nullptr;
  const int64_t n1 = (int64_t)n + 1;
  const int nb = (int)((n1 + SV_T - 1) / SV_T);
  CallScratch scr(st);
  FC_CK(scr.get(&rhs, (size_t)n * sizeof(double)));
  FC_CK(scr.get(&part, (size_t)(nb + 1) * sizeof(double)));
  // grounded system: x(u*) = 0, (I + alpha L) x_V = -1/(n+1) 1
  k_fill<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, -1.0 / (double)n1, rhs);
  FC_LAUNCHED();
  FC_CK(cudaMemsetAsync(x, 0, (size_t)n1 * sizeof(double), st));
  // The right-hand side restricted to V is a multiple of 1, an eigenvector of
  // I + alpha L with eigenvalue 1: unpreconditioned CG reaches it in one step
  // (Jacobi scaling would break that), so the pivot system runs without it.
  const fc_status s = solve_impl(g, alpha_idx, rhs, x, 1, rel_tol, max_iter, iters_out, st, false);
  if (s != FC_OK && s != FC_ENOCONV) return s;
  // shift to the mean-zero gauge of L*^+
  k_partial_sum<<<nb, SV_T, 0, st>>>(n1, x, part);
  fcx::note_launch();
  k_colsum<<<1, SV_T, 0, st>>>(part, nb, part + nb);
  fcx::note_launch();
  k_shift<<<(unsigned)std::min<int64_t>((n1 + 255) / 256, 152 * 8), 256, 0, st>>>(n1, part + nb, x);
  FC_LAUNCHED();
  scr.release();
  FC_CK(cudaStreamSynchronize(st));
  return s;
}

extern "C" fc_status fc_laplacian_solve(fc_graph* g, const double* b, double* x, int32_t n_rhs, double rel_tol,
                                        int32_t max_iter, int32_t* iters_out, void* stream) {
  if (g == nullptr || b == nullptr || x == nullptr || n_rhs < 1 || n_rhs > 65535) {
    set_error("fc_laplacian_solve: bad argument");
    return FC_EINVAL;
  }
  if (g->root < 0) {
    set_error("fc_laplacian_solve: needs a graph from fc_build_rooted (G connected)");
    return FC_EINVAL;
  }
  cudaStream_t st = (cudaStream_t)stream;
  const int32_t n = g->n;
  double* rhs = nullptr;
  double* part = nullptr;
  const int nb = std::max(1, std::min((n + SV_T - 1) / SV_T, 2048 / n_rhs));
  CallScratch scr(st);
  FC_CK(scr.get(&rhs, (size_t)n * n_rhs * sizeof(double)));
  FC_CK(scr.get(&part, (size_t)n_rhs * (nb + 1) * sizeof(double)));
  // b projected onto the range of L (the complement of span(1))
  const fc_status sb = center_columns(n, n_rhs, b, 1, n, rhs, nullptr, part, nb, st);
  if (sb != FC_OK) return sb;
  const fc_status s = solve_impl(g, 0, rhs, x, n_rhs, rel_tol, max_iter, iters_out, st, true, 0.0);
  if (s == FC_OK || s == FC_ENOCONV) {
    // the mean-zero solution: L^+ b
    const fc_status sx = center_columns(n, n_rhs, x, 1, n, x, nullptr, part, nb, st);
    if (sx != FC_OK) return sx;
  }
  scr.release();
  FC_CK(cudaStreamSynchronize(st));
  return s;
}
