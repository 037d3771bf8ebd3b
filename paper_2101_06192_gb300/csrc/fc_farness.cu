// Combination (Algorithm 1's fill step, control variate), forest farness
// (Eq. 3), forest closeness (Def. 2), exact u*-selection probabilities, and
// the top-k ranking (Sec. 6.1).
#include <cooperative_groups.h>

#include <algorithm>
#include <vector>

#include "fc_internal.cuh"

namespace fcx {

// Record msg as the last error and return FC_EINVAL.
static inline fc_status invalid(const char* msg) {
  set_error(msg);
  return FC_EINVAL;
}

constexpr int RED_THREADS = 256;

// p_v = T_v / 2^53 (exact: T_v <= 2^53)
__device__ __forceinline__ double p_from_rowinfo(const uint4& ri) {
  const uint64_t T = (uint64_t)ri.z | ((uint64_t)ri.w << 32);
  return (double)T * 0x1.0p-53;
}

// Pass 1: d_v and per-block partial sums of d (fixed-order tree reduction).
__global__ void k_combine(int32_t n, const uint32_t* __restrict__ R, const uint32_t* __restrict__ C,
                          const float* __restrict__ gpred, const uint4* __restrict__ rinfo,
                          const double* __restrict__ xpiv, double inv_tau, double* __restrict__ diag,
                          double* __restrict__ partial) {
  __shared__ double red[RED_THREADS];
  const int64_t v = (int64_t)blockIdx.x * RED_THREADS + threadIdx.x;
  double d = 0.0;
  if (v < n) {
    d = (double)R[v] * inv_tau;
    if (xpiv != nullptr) {
      // fill step: R/tau - x(u*) + 2 x(v) = diag(L*^+) on V; add back (n+2)/(n+1)^2
      const double n1 = (double)n + 1.0;
      d = d - xpiv[n] + 2.0 * xpiv[v] + ((double)n + 2.0) / (n1 * n1);
    }
    if (C != nullptr) {
      const double p = p_from_rowinfo(rinfo[v]);
      if (p < 1.0) {
        // clip(g, p, 1); a prediction that is not a number counts as p (so
        // every g_pred, NaN included, leaves the estimator unbiased)
        double gg = (double)gpred[v];
        gg = (gg >= p) ? fmin(gg, 1.0) : p;
        const double beta = (1.0 - gg) / (1.0 - p);
        d = d - beta * ((double)C[v] * inv_tau - p);
      }
    }
    diag[v] = d;
  }
  red[threadIdx.x] = d;
  __syncthreads();
  for (int s = RED_THREADS / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}

// Pass 2: single block sums the partials in a fixed order.
__global__ void k_sum_partials(const double* __restrict__ partial, int64_t m, double* __restrict__ out) {
  __shared__ double red[1024];
  double s = 0.0;
  for (int64_t i = threadIdx.x; i < m; i += 1024) s += partial[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int k = 512; k > 0; k >>= 1) {
    if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = red[0];
}

__global__ void k_farness(int32_t n, const double* __restrict__ diag, const double* __restrict__ trace,
                          double* __restrict__ farness, double* __restrict__ closeness) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  const double f = (double)n * diag[v] + *trace - 2.0;  // Eq. 3
  if (farness) farness[v] = f;
  if (closeness) closeness[v] = (double)n / f;         // Def. 2
}

// Batch of graphs: per-graph trace (one block per graph, fixed order) and
// farness with that graph's n and trace.
__global__ void k_seg_trace(const int64_t* __restrict__ voff, const double* __restrict__ diag,
                            double* __restrict__ tr) {
  __shared__ double red[RED_THREADS];
  const int gi = blockIdx.x;
  double s = 0.0;
  for (int64_t v = voff[gi] + threadIdx.x; v < voff[gi + 1]; v += RED_THREADS) s += diag[v];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int k = RED_THREADS / 2; k > 0; k >>= 1) {
    if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
    __syncthreads();
  }
  if (threadIdx.x == 0) tr[gi] = red[0];
}

__global__ void k_farness_seg(int32_t n, const int32_t* __restrict__ gid, const int64_t* __restrict__ voff,
                              const double* __restrict__ diag, const double* __restrict__ tr,
                              double* __restrict__ farness, double* __restrict__ closeness) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  const int32_t gi = gid[v];
  const double ng = (double)(voff[gi + 1] - voff[gi]);
  const double f = ng * diag[v] + tr[gi] - 2.0;  // Eq. 3 within the graph
  if (farness) farness[v] = f;
  if (closeness) closeness[v] = ng / f;          // Def. 2
}

// diag_v = visits[v] / (tau deg*(v)), deg*(v) = fl(1 + fl(alpha d_w(v)))
__global__ void k_visit_diag(int32_t n, const unsigned long long* __restrict__ visits, double alpha_s,
                             const double* __restrict__ alpha_v, const double* __restrict__ dw, double tau,
                             double* __restrict__ diag) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  const double a = alpha_v ? alpha_v[v] : alpha_s;
  diag[v] = __ddiv_rn((double)visits[v], __dmul_rn(tau, deg_star(a, dw[v])));
}

__global__ void k_p_root(int32_t n, const uint4* __restrict__ rinfo, double* __restrict__ p) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n) p[v] = p_from_rowinfo(rinfo[v]);
}

// ---------------------------------------------------------------------------
// top-k: the k smallest (key, id) pairs, key = order-preserving 64-bit image of
// diag.  For k <= TS_K a radix selection (k_ts_select) finds the pair of rank k
// digit by digit and stops as soon as at most TS_CAP pairs share its prefix;
// the pairs below the prefix and those on it, at most TS_N, are sorted by one
// block (k_ts_sort).  Larger k: stable LSD radix sort of all pairs (inputs in id
// order, so equal keys keep ascending ids).  Bound by launches and passes over
// diag: measured on GB300 for k = 10 against the sort, whole calls: n = 1000 270 ->
// 53 us, n = 2^20 371 -> 63 us, n = 2^22 (R-MAT) 580 -> 309 us.
// ---------------------------------------------------------------------------
constexpr int TK_TILE = 1024;

// Order-preserving key: -0.0 and +0.0 compare equal (ties then go by id) and
// every NaN sorts after +inf.
__device__ __forceinline__ uint64_t ordered_key(double d) {
  if (d == 0.0) d = 0.0;
  if (isnan(d)) return ~0ull;
  uint64_t u = (uint64_t)__double_as_longlong(d);
  return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}

__global__ void k_tk_init(int32_t n, const double* __restrict__ diag, uint64_t* __restrict__ keys,
                          int32_t* __restrict__ vals) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n) {
    keys[v] = ordered_key(diag[v]);
    vals[v] = (int32_t)v;
  }
}

__global__ void k_tk_hist(int32_t n, const uint64_t* __restrict__ keys, int shift, uint32_t* __restrict__ hist,
                          int32_t nblk) {
  __shared__ uint32_t cnt[256];
  const int lane = threadIdx.x;
  for (int d = lane; d < 256; d += 32) cnt[d] = 0;
  __syncwarp();
  const int64_t base = (int64_t)blockIdx.x * TK_TILE;
  for (int c = 0; c < TK_TILE / 32; ++c) {
    const int64_t i = base + c * 32 + lane;
    if (i < n) atomicAdd(&cnt[(uint32_t)(keys[i] >> shift) & 255u], 1u);
  }
  __syncwarp();
  for (int d = lane; d < 256; d += 32) hist[(int64_t)d * nblk + blockIdx.x] = cnt[d];
}

__global__ void k_tk_scatter(int32_t n, const uint64_t* __restrict__ kin, const int32_t* __restrict__ vin,
                             uint64_t* __restrict__ kout, int32_t* __restrict__ vout, int shift,
                             const uint32_t* __restrict__ offs, int32_t nblk) {
  __shared__ uint32_t run[256];
  const int lane = threadIdx.x;
  for (int d = lane; d < 256; d += 32) run[d] = offs[(int64_t)d * nblk + blockIdx.x];
  __syncwarp();
  const int64_t base = (int64_t)blockIdx.x * TK_TILE;
  const unsigned lt = (1u << lane) - 1u;
  for (int c = 0; c < TK_TILE / 32; ++c) {
    const int64_t i = base + c * 32 + lane;
    const bool valid = i < n;
    uint64_t key = 0;
    int32_t val = 0;
    uint32_t d = 256u + lane;
    if (valid) {
      key = kin[i];
      val = vin[i];
      d = (uint32_t)(key >> shift) & 255u;
    }
    const unsigned peers = __match_any_sync(0xffffffffu, d);
    const uint32_t rank = __popc(peers & lt);
    if (valid) {
      const uint32_t pos = run[d] + rank;
      kout[pos] = key;
      vout[pos] = val;
    }
    __syncwarp();
    if (valid && lane == __ffs(peers) - 1) run[d] += __popc(peers);
    __syncwarp();
  }
}

constexpr int TS_T = 512;
constexpr int TS_BITS = 11;
constexpr int TS_BINS = 1 << TS_BITS;
constexpr int TS_PASSES = 9;   // key digits 11 x 5 + 9, id digits 11 + 11 + 9 (31 bits: every id)
constexpr int TS_CAP = 1024;   // pairs on the prefix that end the selection
constexpr int TS_N = 4096;     // pairs sorted by one block
constexpr int TS_K = TS_N - TS_CAP;

// digit of pass p of a pair, and whether the pair lies on the prefix of the
// passes before (same higher digits)
struct TSPrefix {
  uint64_t key;  // digits of the key so far, in place
  uint32_t id;
};
__device__ __forceinline__ int ts_shift(int p) { return p < 5 ? 53 - 11 * p : p == 5 ? 0 : p == 6 ? 20 : p == 7 ? 9 : 0; }
__device__ __forceinline__ int ts_bits(int p) { return p == 5 || p == 8 ? 9 : TS_BITS; }
__device__ __forceinline__ uint32_t ts_digit(uint64_t key, uint32_t id, int p) {
  const uint64_t x = p < 6 ? key : (uint64_t)id;
  return (uint32_t)(x >> ts_shift(p)) & ((1u << ts_bits(p)) - 1u);
}
// -1 / 0 / +1: the pair is below / on / above the prefix of p digits
__device__ __forceinline__ int ts_side(uint64_t key, uint32_t id, const TSPrefix& f, int p) {
  if (p == 0) return 0;
  const int q = p < 6 ? p : 6;  // key digits known
  const int sh = ts_shift(q - 1);
  const uint64_t a = key >> sh, b = f.key >> sh;
  if (a != b) return a < b ? -1 : 1;
  if (p <= 6) return 0;
  const int si = ts_shift(p - 1);
  const uint32_t c = id >> si, d = f.id >> si;
  return c == d ? 0 : c < d ? -1 : 1;
}

// hist: [TS_PASSES][TS_BINS] zeroed; count: zeroed; buf: the collected pairs.
// Cooperative: every block reads the finished histogram of a pass and takes
// the same decision.
__global__ void __launch_bounds__(TS_T) k_ts_select(int32_t n, const double* __restrict__ diag, int32_t k,
                                                    uint32_t* __restrict__ hist, uint32_t* __restrict__ count,
                                                    uint64_t* __restrict__ bkey, int32_t* __restrict__ bid) {
  cooperative_groups::grid_group grid = cooperative_groups::this_grid();
  __shared__ uint32_t h[TS_BINS];
  __shared__ uint32_t wsum[TS_T / 32];
  __shared__ uint32_t sh_digit, sh_below, sh_on;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t gtid = (int64_t)blockIdx.x * TS_T + threadIdx.x, gstride = (int64_t)gridDim.x * TS_T;
  TSPrefix f{0, 0};
  uint32_t rem = (uint32_t)k;  // rank of the wanted pair among those on the prefix
  uint32_t on = (uint32_t)n;   // pairs on the prefix
  int p = 0;
  for (; on > (uint32_t)TS_CAP && p < TS_PASSES; ++p) {
    for (int i = threadIdx.x; i < TS_BINS; i += TS_T) h[i] = 0u;
    __syncthreads();
    for (int64_t i = gtid; i < n; i += gstride) {
      const uint64_t key = ordered_key(diag[i]);
      const bool in = ts_side(key, (uint32_t)i, f, p) == 0;
      // values crowd on few leading digits: one atomic per distinct digit of the warp
      const unsigned act = __activemask();
      const uint32_t d = in ? ts_digit(key, (uint32_t)i, p) : (uint32_t)TS_BINS;
      const unsigned peers = __match_any_sync(act, d);
      if (in && lane == __ffs(peers) - 1) atomicAdd(&h[d], (uint32_t)__popc(peers));
    }
    __syncthreads();
    for (int i = threadIdx.x; i < TS_BINS; i += TS_T)
      if (h[i]) atomicAdd(&hist[p * TS_BINS + i], h[i]);
    grid.sync();
    // the digit that holds rank rem: an exclusive scan of the bins, four per thread
    uint32_t c[TS_BINS / TS_T], s = 0;
#pragma unroll
    for (int q = 0; q < TS_BINS / TS_T; ++q) {
      c[q] = __ldcg(&hist[p * TS_BINS + threadIdx.x * (TS_BINS / TS_T) + q]);
      s += c[q];
    }
    uint32_t inc = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[wid] = inc;
    __syncthreads();
    uint32_t below = inc - s;
    for (int q = 0; q < wid; ++q) below += wsum[q];
#pragma unroll
    for (int q = 0; q < TS_BINS / TS_T; ++q) {
      if (below < rem && rem <= below + c[q]) {  // exactly one thread and digit
        sh_digit = threadIdx.x * (TS_BINS / TS_T) + q;
        sh_below = below;
        sh_on = c[q];
      }
      below += c[q];
    }
    __syncthreads();
    if (p < 6) f.key |= (uint64_t)sh_digit << ts_shift(p);
    else f.id |= sh_digit << ts_shift(p);
    rem -= sh_below;
    on = sh_on;
    __syncthreads();  // read before the next pass writes them
  }
  for (int64_t i = gtid; i < n; i += gstride) {
    const uint64_t key = ordered_key(diag[i]);
    if (ts_side(key, (uint32_t)i, f, p) <= 0) {
      const uint32_t at = atomicAdd(count, 1u);  // at most k - rem + on <= TS_N
      bkey[at] = key;
      bid[at] = (int32_t)i;
    }
  }
}

// bitonic sort of the collected pairs by (key, id); the first k ids
__global__ void __launch_bounds__(1024) k_ts_sort(const uint32_t* __restrict__ count, const uint64_t* __restrict__ bkey,
                                                  const int32_t* __restrict__ bid, int32_t k,
                                                  int32_t* __restrict__ idx_out) {
  __shared__ uint64_t key[TS_N];
  __shared__ int32_t id[TS_N];
  const int cnt = (int)*count;
  int m = 32;
  while (m < cnt) m <<= 1;
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    key[i] = i < cnt ? bkey[i] : ~0ull;
    id[i] = i < cnt ? bid[i] : INT32_MAX;  // after every real pair
  }
  __syncthreads();
  for (int s = 2; s <= m; s <<= 1)
    for (int j = s >> 1; j > 0; j >>= 1) {
      for (int t = threadIdx.x; t < m / 2; t += blockDim.x) {
        const int i = 2 * t - (t & (j - 1)), l = i + j;
        const bool up = (i & s) == 0;
        const uint64_t a = key[i], b = key[l];
        const int32_t ia = id[i], ib = id[l];
        const bool gt = a > b || (a == b && ia > ib);
        if (gt == up) {
          key[i] = b;
          key[l] = a;
          id[i] = ib;
          id[l] = ia;
        }
      }
      __syncthreads();
    }
  for (int i = threadIdx.x; i < k; i += blockDim.x) idx_out[i] = id[i];
}

// per-block sums of diag in the same fixed tree order as k_combine's
__global__ void k_block_sums(int32_t n, const double* __restrict__ diag, double* __restrict__ partial) {
  __shared__ double red[RED_THREADS];
  const int64_t v = (int64_t)blockIdx.x * RED_THREADS + threadIdx.x;
  red[threadIdx.x] = v < n ? diag[v] : 0.0;
  __syncthreads();
  for (int s = RED_THREADS / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}

}  // namespace fcx

using namespace fcx;

extern "C" fc_status fc_forest_farness(fc_graph* g, int32_t alpha_idx, const uint32_t* R, const uint32_t* C,
                                       const float* g_pred, const double* x_pivot, int64_t tau,
                                       double* diag_out, double* farness_out, double* closeness_out,
                                       void* stream) {
  if (g == nullptr || R == nullptr || diag_out == nullptr || tau < 1 || alpha_idx < 0 ||
      alpha_idx >= g->n_alpha || ((C == nullptr) != (g_pred == nullptr))) {
    set_error("fc_forest_farness: bad argument");
    return FC_EINVAL;
  }
  cudaStream_t st = (cudaStream_t)stream;
  const int32_t n = g->n;
  const int64_t nb = (n + RED_THREADS - 1) / RED_THREADS;
  double* partial = nullptr;
  FC_CK(cudaMallocAsync((void**)&partial, (nb + 1) * sizeof(double), st));
  const uint4* rinfo = g->rowinfo + (size_t)alpha_idx * n;
  k_combine<<<(unsigned)nb, RED_THREADS, 0, st>>>(n, R, C, g_pred, rinfo, x_pivot, 1.0 / (double)tau, diag_out,
                                                  partial);
  FC_LAUNCHED();
  if (g->num_graphs > 0) {
    double* tr = nullptr;
    FC_CK(cudaMallocAsync((void**)&tr, (size_t)g->num_graphs * sizeof(double), st));
    k_seg_trace<<<g->num_graphs, RED_THREADS, 0, st>>>(g->voff, diag_out, tr);
    FC_LAUNCHED();
    if (farness_out || closeness_out) {
      k_farness_seg<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, g->gid, g->voff, diag_out, tr, farness_out,
                                                                 closeness_out);
      FC_LAUNCHED();
    }
    FC_CK(cudaFreeAsync(tr, st));
    FC_CK(cudaFreeAsync(partial, st));
    return FC_OK;
  }
  k_sum_partials<<<1, 1024, 0, st>>>(partial, nb, partial + nb);
  FC_LAUNCHED();
  if (farness_out || closeness_out) {
    k_farness<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, diag_out, partial + nb, farness_out, closeness_out);
    FC_LAUNCHED();
  }
  FC_CK(cudaFreeAsync(partial, st));
  return FC_OK;
}

extern "C" fc_status fc_farness_from_diag(fc_graph* g, const double* diag, double* farness_out,
                                          double* closeness_out, void* stream) {
  if (g == nullptr || diag == nullptr) {
    set_error("fc_farness_from_diag: bad argument");
    return FC_EINVAL;
  }
  if (farness_out == nullptr && closeness_out == nullptr) return FC_OK;
  cudaStream_t st = (cudaStream_t)stream;
  const int32_t n = g->n;
  if (g->num_graphs > 0) {
    double* tr = nullptr;
    FC_CK(cudaMallocAsync((void**)&tr, (size_t)g->num_graphs * sizeof(double), st));
    k_seg_trace<<<g->num_graphs, RED_THREADS, 0, st>>>(g->voff, diag, tr);
    FC_LAUNCHED();
    k_farness_seg<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, g->gid, g->voff, diag, tr, farness_out,
                                                               closeness_out);
    FC_LAUNCHED();
    FC_CK(cudaFreeAsync(tr, st));
    return FC_OK;
  }
  const int64_t nb = (n + RED_THREADS - 1) / RED_THREADS;
  double* partial = nullptr;
  FC_CK(cudaMallocAsync((void**)&partial, (nb + 1) * sizeof(double), st));
  k_block_sums<<<(unsigned)nb, RED_THREADS, 0, st>>>(n, diag, partial);
  FC_LAUNCHED();
  k_sum_partials<<<1, 1024, 0, st>>>(partial, nb, partial + nb);
  FC_LAUNCHED();
  k_farness<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, diag, partial + nb, farness_out, closeness_out);
  FC_LAUNCHED();
  FC_CK(cudaFreeAsync(partial, st));
  return FC_OK;
}

extern "C" fc_status fc_p_root(fc_graph* g, int32_t alpha_idx, double* p_out, void* stream) {
  if (g == nullptr || p_out == nullptr || alpha_idx < 0 || alpha_idx >= g->n_alpha)
    return fcx::invalid("fc_p_root: bad argument");
  cudaStream_t st = (cudaStream_t)stream;
  k_p_root<<<(unsigned)((g->n + 255) / 256), 256, 0, st>>>(g->n, g->rowinfo + (size_t)alpha_idx * g->n, p_out);
  FC_LAUNCHED();
  return FC_OK;
}

extern "C" fc_status fc_top_k(const double* diag, int32_t n, int32_t k, int32_t* idx_out, void* stream) {
  if (diag == nullptr || idx_out == nullptr || n < 1 || k < 1 || k > n) {
    set_error("fc_top_k: bad argument");
    return FC_EINVAL;
  }
  cudaStream_t st = (cudaStream_t)stream;
  if (k <= TS_K) {
    int dev = 0, nsm = 0, per_sm = 0, coop = 0;
    FC_CK(cudaGetDevice(&dev));
    FC_CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    FC_CK(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
    FC_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_ts_select, TS_T, 0));
    if (coop && per_sm > 0) {
      uint64_t* bkey = nullptr;
      const size_t hb = (size_t)TS_PASSES * TS_BINS * 4 + 16;
      FC_CK(cudaMallocAsync((void**)&bkey, (size_t)TS_N * 12 + hb, st));
      int32_t* bid = (int32_t*)(bkey + TS_N);
      uint32_t* hist = (uint32_t*)(bid + TS_N);
      uint32_t* count = hist + TS_PASSES * TS_BINS;
      FC_CK(cudaMemsetAsync(hist, 0, hb, st));
      // blocks: four values per thread, at most two per SM (the barriers of few blocks are quicker)
      int blocks = (int)std::min<int64_t>(((int64_t)n + 4 * TS_T - 1) / (4 * TS_T), (int64_t)std::min(per_sm, 2) * nsm);
      void* args[] = {&n, &diag, &k, &hist, &count, &bkey, &bid};
      FC_CK(cudaLaunchCooperativeKernel((const void*)k_ts_select, dim3(blocks), dim3(TS_T), args, 0, st));
      FC_LAUNCHED();
      k_ts_sort<<<1, 1024, 0, st>>>(count, bkey, bid, k, idx_out);
      FC_LAUNCHED();
      FC_CK(cudaFreeAsync(bkey, st));
      FC_CK(cudaStreamSynchronize(st));
      return FC_OK;
    }
  }
  const int32_t nblk = (n + TK_TILE - 1) / TK_TILE;
  const int64_t hlen = (int64_t)256 * nblk;
  uint64_t *k0 = nullptr, *k1 = nullptr;
  int32_t *v0 = nullptr, *v1 = nullptr;
  uint32_t *hist = nullptr, *offs = nullptr;
  FC_CK(cudaMallocAsync((void**)&k0, (size_t)n * 8, st));
  FC_CK(cudaMallocAsync((void**)&k1, (size_t)n * 8, st));
  FC_CK(cudaMallocAsync((void**)&v0, (size_t)n * 4, st));
  FC_CK(cudaMallocAsync((void**)&v1, (size_t)n * 4, st));
  FC_CK(cudaMallocAsync((void**)&hist, (size_t)hlen * 4, st));
  FC_CK(cudaMallocAsync((void**)&offs, (size_t)hlen * 4, st));
  k_tk_init<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, diag, k0, v0);
  FC_LAUNCHED();
  uint64_t* kin = k0;
  uint64_t* kout = k1;
  int32_t* vin = v0;
  int32_t* vout = v1;
  for (int pass = 0; pass < 8; ++pass) {
    k_tk_hist<<<nblk, 32, 0, st>>>(n, kin, 8 * pass, hist, nblk);
    FC_LAUNCHED();
    const fc_status r = exclusive_scan(hist, offs, hlen, st);
    if (r != FC_OK) return r;
    k_tk_scatter<<<nblk, 32, 0, st>>>(n, kin, vin, kout, vout, 8 * pass, offs, nblk);
    FC_LAUNCHED();
    std::swap(kin, kout);
    std::swap(vin, vout);
  }
  FC_CK(cudaMemcpyAsync(idx_out, vin, (size_t)k * 4, cudaMemcpyDeviceToDevice, st));
  FC_CK(cudaFreeAsync(k0, st));
  FC_CK(cudaFreeAsync(k1, st));
  FC_CK(cudaFreeAsync(v0, st));
  FC_CK(cudaFreeAsync(v1, st));
  FC_CK(cudaFreeAsync(hist, st));
  FC_CK(cudaFreeAsync(offs, st));
  FC_CK(cudaStreamSynchronize(st));
  return FC_OK;
}

// ---------------------------------------------------------------------------
// Allocation-free variant of fc_forest_farness.  The per-block partial sums
// and the trace live in a file-scope device array instead of stream-ordered
// pool memory.  Host code must not pass the array's name to a kernel (on the
// host it is only a stand-in symbol), so its device address on the current
// device is looked up with cudaGetSymbolAddress at every call (a host-side
// lookup; nothing cached, so a reset device or a reloaded module is no issue).
// ---------------------------------------------------------------------------
namespace fcx {
constexpr int32_t NOALLOC_MAX_N = 1 << 22;
constexpr int64_t NOALLOC_MAX_BLOCKS = (NOALLOC_MAX_N + RED_THREADS - 1) / RED_THREADS;
static __device__ __align__(256) double g_noalloc_partials[NOALLOC_MAX_BLOCKS + 1];

static fc_status noalloc_scratch(double** out) {
  void* p = nullptr;
  FC_CK(cudaGetSymbolAddress(&p, g_noalloc_partials));
  *out = (double*)p;
  return FC_OK;
}
}  // namespace fcx

extern "C" fc_status fc_forest_farness_noalloc(fc_graph* g, int32_t alpha_idx, const uint32_t* R,
                                               const uint32_t* C, const float* g_pred, const double* x_pivot,
                                               int64_t tau, double* diag_out, double* farness_out,
                                               double* closeness_out, void* stream) {
  if (g == nullptr || R == nullptr || diag_out == nullptr || tau < 1 || alpha_idx < 0 ||
      alpha_idx >= g->n_alpha || ((C == nullptr) != (g_pred == nullptr))) {
    set_error("fc_forest_farness_noalloc: bad argument");
    return FC_EINVAL;
  }
  if (g->num_graphs > 0) {
    set_error("fc_forest_farness_noalloc: batches of graphs need per-graph traces; use fc_forest_farness");
    return FC_EINVAL;
  }
  if (g->n > NOALLOC_MAX_N) {
    set_error("fc_forest_farness_noalloc: n exceeds the fixed scratch capacity of 4194304 vertices; "
              "use fc_forest_farness");
    return FC_EINVAL;
  }
  int dev = -1;
  FC_CK(cudaGetDevice(&dev));
  if (dev != g->device) {
    set_error("fc_forest_farness_noalloc: the graph's device is not the current device");
    return FC_EINVAL;
  }
  double* partial = nullptr;
  const fc_status s = noalloc_scratch(&partial);
  if (s != FC_OK) return s;
  cudaStream_t st = (cudaStream_t)stream;
  const int32_t n = g->n;
  const int64_t nb = (n + RED_THREADS - 1) / RED_THREADS;
  const uint4* rinfo = g->rowinfo + (size_t)alpha_idx * n;
  // k_combine writes partial[0, nb) and k_sum_partials writes partial[nb]
  // before anything reads them, so no clearing is needed between calls.
  k_combine<<<(unsigned)nb, RED_THREADS, 0, st>>>(n, R, C, g_pred, rinfo, x_pivot, 1.0 / (double)tau, diag_out,
                                                  partial);
  FC_LAUNCHED();
  k_sum_partials<<<1, 1024, 0, st>>>(partial, nb, partial + nb);
  FC_LAUNCHED();
  if (farness_out || closeness_out) {
    k_farness<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, diag_out, partial + nb, farness_out, closeness_out);
    FC_LAUNCHED();
  }
  return FC_OK;
}

extern "C" fc_status fc_visit_diag(fc_graph* g, int32_t alpha_idx, const uint64_t* visits, int64_t tau,
                                   double* diag_out, void* stream) {
  if (g == nullptr || visits == nullptr || diag_out == nullptr || tau < 1 || alpha_idx < 0 ||
      alpha_idx >= g->n_alpha || g->root >= 0) {
    set_error("fc_visit_diag: bad argument (a graph from fc_build_augmented or fc_build_batch)");
    return FC_EINVAL;
  }
  cudaStream_t st = (cudaStream_t)stream;
  const int32_t n = g->n;
  k_visit_diag<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(
      n, (const unsigned long long*)visits + (size_t)alpha_idx * n, g->alphas[alpha_idx],
      g->num_graphs > 0 ? g->alpha_v : nullptr, g->dw, (double)tau, diag_out);
  FC_LAUNCHED();
  return FC_OK;
}
