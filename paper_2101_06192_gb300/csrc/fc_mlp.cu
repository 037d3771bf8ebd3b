// Learned control variate (not in the paper): a two-layer perceptron that
// predicts g_v ~ Omega_vv from local features of v; the prediction only sets
// the control-variate coefficient beta_v = (1 - g_v) / (1 - p_v), so the
// estimator stays unbiased whatever the network outputs.
//
//   features  x = (log(1 + deg), log(1 + alpha d_w), log(1 + sum_{u in N(v)} deg(u)), log(alpha))
//   network   h = relu(W1 x + b1) (128 units), z = w2 . h + b2,
//             g = p + (1 - p) sigmoid(z)
//   loss      mean over vertices of (g - y)^2
//   optimiser Adam (Kingma & Ba) with bias correction
//
// Parameters: one FP32 master vector of MLP_NPARAM floats laid out as
// W1[128][4], b1[128], w2[128], b2.  Every kernel reads them rounded to BF16
// (round to nearest even) and accumulates in FP32.  The hidden layer has K = 4
// and the output layer N = 1, so these are per-vertex dot products on the
// CUDA cores, bound by issue slots: 5 FMAs, a maximum and the weights' loads per
// vertex and hidden unit, against a 16-byte feature row per vertex.  So a thread
// of the forward pass takes up to eight vertices per load of a unit's weights, and a
// lane of the gradient pass four units per load of a vertex's features.
// Measured on GB300 (whole calls, against one vertex and one unit): forward pass
// n = 2^22 190 -> 139 us; loss and gradient n = 2^22 475 -> 397, 2^18 53 -> 42.
// Packed FP32 pairs (fma.rn.f32x2) issued as many instructions: 200 us.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

#include "fc_internal.cuh"

namespace fcx {

constexpr int HID = 128;
constexpr int NF = 4;
constexpr int OFF_W1 = 0, OFF_B1 = HID * NF, OFF_W2 = OFF_B1 + HID, OFF_B2 = OFF_W2 + HID;
constexpr int NPARAM = OFF_B2 + 1;  // 769
constexpr int MLP_T = 128;          // threads per block (one hidden unit each in the gradient pass)

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// p = T 2^-53 rounded to FP32.  T <= 2^53, so this is the FP64 value rounded
// once (the FP64 pipe would be the cost: two results per clock and SM).
__device__ __forceinline__ float p_of(const uint4& ri) {
  const uint64_t T = (uint64_t)ri.z | ((uint64_t)ri.w << 32);
  return __ull2float_rn(T) * 0x1.0p-53f;
}

// Sum over neighbours of their degree, s2[v] = sum over w in N(v) of deg(w).
// A block takes consecutive tiles of NDS_TILE CSR entries whatever rows they
// belong to: every thread has NDS_U neighbour gathers in flight, the tile's
// prefix sums go to shared memory, and a thread per row of the tile takes the
// difference over its entries.  Rows inside the tile are stored, rows that
// cross tiles add their parts (integers: any order gives the same result).
// The gathers of the next tile and the column indices of the one after it are
// under way meanwhile; the first tile's first row comes from a 32-way search,
// the later ones' from the tile before.  Bound by the gathers of deg.  (Before:
// a warp walked 1024 entries in 32 dependent steps.  Features on GB300, whole
// calls: R-MAT n = 2^16 37 -> 25 us, 2^18 64 -> 49, 2^22 786 -> 606.)
constexpr int NDS_T = 256;
constexpr int NDS_U = 8;
constexpr int NDS_TILE = NDS_T * NDS_U;
constexpr unsigned NDS_FULL = 0xffffffffu;
__device__ __forceinline__ int nds_pad(int i) { return i + (i >> 3); }  // eight per thread without bank conflicts

__global__ void __launch_bounds__(NDS_T, 6) k_nbr_deg_sum(int32_t n, int64_t nnz, const int64_t* __restrict__ rowptr,
                                                          const int32_t* __restrict__ colidx,
                                                          const int32_t* __restrict__ deg, int64_t per,
                                                          unsigned long long* __restrict__ s2) {
  __shared__ unsigned long long P[NDS_TILE + NDS_TILE / 8 + 1];  // exclusive prefix sums, padded
  __shared__ __align__(16) uint32_t val[NDS_TILE];
  __shared__ unsigned long long wsum[NDS_T / 32];
  __shared__ int32_t first[2];  // first row of the tile, by the tile's parity
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t b0 = (int64_t)blockIdx.x * per * NDS_TILE;
  const int64_t b1 = b0 + per * NDS_TILE < nnz ? b0 + per * NDS_TILE : nnz;  // this block's entries
  int32_t c[NDS_U];
  uint32_t d[NDS_U];
  auto cols = [&](int64_t e0) {
#pragma unroll
    for (int k = 0; k < NDS_U; ++k) {
      const int64_t e = e0 + k * NDS_T + threadIdx.x;
      c[k] = e < b1 ? __ldcs(colidx + e) : -1;
    }
  };
  auto gather = [&]() {
#pragma unroll
    for (int k = 0; k < NDS_U; ++k) d[k] = c[k] >= 0 ? (uint32_t)__ldg(deg + c[k]) : 0u;
  };
  cols(b0);
  gather();
  cols(b0 + NDS_TILE);
  if (wid == 0) {  // the last row v with rowptr[v] <= b0: rowptr[lo] <= b0 < rowptr[hi]
    int32_t lo = 0, hi = n;
    while (hi - lo > 1) {
      const int32_t step = hi - lo >= 64 ? (hi - lo) / 32 : 1;
      const int64_t x = (int64_t)lo + (int64_t)step * (lane + 1);
      const int cnt = __popc(__ballot_sync(NDS_FULL, x < hi && rowptr[x < hi ? x : lo] <= b0));
      lo += step * cnt;
      if (cnt < 32 && hi - lo > step) hi = lo + step;
    }
    if (lane == 0) first[0] = lo;
  }
  int par = 0;
  for (int64_t e0 = b0; e0 < b1; e0 += NDS_TILE, par ^= 1) {
    const int64_t e1 = e0 + NDS_TILE < b1 ? e0 + NDS_TILE : b1;
#pragma unroll
    for (int k = 0; k < NDS_U; ++k) val[k * NDS_T + threadIdx.x] = d[k];
    gather();
    cols(e0 + 2 * NDS_TILE);
    __syncthreads();
    unsigned long long x[NDS_U], s = 0;
    const uint4* v4 = reinterpret_cast<const uint4*>(val + threadIdx.x * NDS_U);
    const uint4 va = v4[0], vb = v4[1];
    const uint32_t v[NDS_U] = {va.x, va.y, va.z, va.w, vb.x, vb.y, vb.z, vb.w};
#pragma unroll
    for (int k = 0; k < NDS_U; ++k) {
      x[k] = s;
      s += v[k];
    }
    unsigned long long inc = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(NDS_FULL, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[wid] = inc;
    __syncthreads();
    unsigned long long base = inc - s;
    for (int q = 0; q < wid; ++q) base += wsum[q];
#pragma unroll
    for (int k = 0; k < NDS_U; ++k) P[nds_pad(threadIdx.x * NDS_U + k)] = base + x[k];
    if (threadIdx.x == NDS_T - 1) P[nds_pad(NDS_TILE)] = base + s;
    __syncthreads();
    for (int64_t r = first[par] + (int64_t)threadIdx.x; r < n; r += NDS_T) {
      const int64_t r0 = rowptr[r], r1 = rowptr[r + 1];
      if (r0 >= e1) break;
      if (r1 >= e1) first[par ^ 1] = (int32_t)r;  // one row: the last that starts before e1
      const int64_t a0 = r0 > e0 ? r0 : e0, a1 = r1 < e1 ? r1 : e1;
      if (a1 <= a0) continue;  // an empty row (zero already), or one that ended with the tile before
      const unsigned long long sum = P[nds_pad((int)(a1 - e0))] - P[nds_pad((int)(a0 - e0))];
      if (a0 == r0 && a1 == r1) s2[r] = sum;
      else atomicAdd(&s2[r], sum);
    }
  }
}

__global__ void k_features(int32_t n, double alpha_s, const double* __restrict__ alpha_v,
                           const int32_t* __restrict__ deg, const double* __restrict__ dw,
                           const unsigned long long* __restrict__ s2, float4* __restrict__ X) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    // FP32 logarithms (GB300's FP64 rate made the FP64 ones the cost of the
    // feature pass); the inputs are rounded to FP32 first
    const double alpha = alpha_v ? alpha_v[v] : alpha_s;
    X[v] = make_float4(log1pf((float)deg[v]), log1pf((float)(alpha * dw[v])), log1pf((float)s2[v]),
                       logf((float)alpha));
  }
}

// The (BF16-valued) weights of a hidden unit: two loads
struct __align__(16) Unit {
  float4 w;      // W1[j]
  float b, w2;   // b1[j], w2[j]
  float pad[2];
};
__device__ __forceinline__ void load_params(const float* __restrict__ params, Unit* su) {
  for (int j = threadIdx.x; j < HID; j += blockDim.x) {
    const float* w = params + OFF_W1 + j * NF;
    su[j].w = make_float4(bf16r(w[0]), bf16r(w[1]), bf16r(w[2]), bf16r(w[3]));
    su[j].b = bf16r(params[OFF_B1 + j]);
    su[j].w2 = bf16r(params[OFF_W2 + j]);
  }
  __syncthreads();
}

// W1[j] x + b1[j]
__device__ __forceinline__ float mlp_pre(const float4& w, float b, const float4& x) {
  float pre = fmaf(w.x, x.x, b);
  pre = fmaf(w.y, x.y, pre);
  pre = fmaf(w.z, x.z, pre);
  return fmaf(w.w, x.w, pre);
}

// z = w2 . relu(W1 x + b1) + b2 of NV vertices
template <int NV>
__device__ __forceinline__ void mlp_z(const Unit* su, float b2, const float4 (&x)[NV], float (&z)[NV]) {
#pragma unroll
  for (int i = 0; i < NV; ++i) z[i] = b2;
#pragma unroll 4
  for (int j = 0; j < HID; ++j) {
    const float4 w = su[j].w;
    const float2 u = *reinterpret_cast<const float2*>(&su[j].b);
#pragma unroll
    for (int i = 0; i < NV; ++i) z[i] = fmaf(u.y, fmaxf(mlp_pre(w, u.x, x[i]), 0.0f), z[i]);
  }
}

__device__ __forceinline__ float mlp_g(float z, const uint4& ri) {
  const float s = 1.0f / (1.0f + expf(-z));
  const float p = p_of(ri);
  return p + (1.0f - p) * s;
}

// NV vertices per thread
template <int NV>
__global__ void __launch_bounds__(MLP_T) k_mlp_forward(int32_t n, const float4* __restrict__ X,
                                                       const uint4* __restrict__ rinfo,
                                                       const float* __restrict__ params, float* __restrict__ gout) {
  __shared__ Unit su[HID];
  load_params(params, su);
  const float b2 = bf16r(params[OFF_B2]);
  const int64_t step = NV * MLP_T;
  for (int64_t base = blockIdx.x * step; base < n; base += gridDim.x * step) {
    float4 x[NV];
    float z[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int64_t v = base + i * MLP_T + threadIdx.x;
      x[i] = v < n ? X[v] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    mlp_z<NV>(su, b2, x, z);
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int64_t v = base + i * MLP_T + threadIdx.x;
      if (v < n) gout[v] = mlp_g(z[i], rinfo[v]);
    }
  }
}

// Loss and gradient, per-block partials (fixed order, deterministic).
// Pass over tiles of NV MLP_T vertices: a thread runs the forward pass of NV
// vertices and their dL/dz; then warp w takes a quarter of the tile's vertices,
// each lane the gradient of four hidden units, so that a load of a vertex's
// features serves four units; the warps have sums of their own, added at the
// end.  w2[j], the same factor in every
// term of the hidden layer's gradient, is multiplied once at the end.
constexpr int MLP_W = MLP_T / 32;
constexpr int MLP_UL = HID / 32;  // hidden units per lane
constexpr int GRAD_V = NF + 2;    // sums per hidden unit
static_assert(HID == MLP_T, "a thread per hidden unit writes the partials");
template <int NV>
__global__ void __launch_bounds__(MLP_T) k_mlp_grad(int32_t n, const float4* __restrict__ X,
                                                    const uint4* __restrict__ rinfo, const float* __restrict__ y,
                                                    const float* __restrict__ params, float inv_n,
                                                    float* __restrict__ gpart, double* __restrict__ lpart) {
  constexpr int TILE = NV * MLP_T;
  __shared__ Unit su[HID];
  __shared__ float4 sx[TILE];
  __shared__ float sdz[TILE];
  __shared__ float sg[MLP_W][GRAD_V][HID];
  __shared__ float sb[MLP_W];
  __shared__ double sl[MLP_T];
  load_params(params, su);
  const float b2 = bf16r(params[OFF_B2]);
  const int j = threadIdx.x, lane = j & 31, wid = j >> 5;
  float4 w[MLP_UL], gW[MLP_UL];
  float ub[MLP_UL], gb1[MLP_UL], gw2[MLP_UL];
#pragma unroll
  for (int q = 0; q < MLP_UL; ++q) {
    w[q] = su[lane + 32 * q].w;
    ub[q] = su[lane + 32 * q].b;
    gW[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    gb1[q] = gw2[q] = 0.f;
  }
  float gb2 = 0.f;
  double lsum = 0.0;
  for (int64_t base = (int64_t)blockIdx.x * TILE; base < n; base += (int64_t)gridDim.x * TILE) {
    float4 x[NV];
    float z[NV];
    bool fin = true;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int64_t v = base + i * MLP_T + j;
      x[i] = v < n ? X[v] : make_float4(0.f, 0.f, 0.f, 0.f);
      fin = fin && isfinite(x[i].x) && isfinite(x[i].y) && isfinite(x[i].z) && isfinite(x[i].w);
    }
    mlp_z<NV>(su, b2, x, z);
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int64_t v = base + i * MLP_T + j;
      float dz = 0.f;
      if (v < n) {
        const float s = 1.0f / (1.0f + expf(-z[i]));
        const float p = p_of(rinfo[v]);
        const float g = p + (1.0f - p) * s;
        const float r = g - y[v];
        lsum += (double)r * (double)r;
        dz = 2.0f * r * inv_n * (1.0f - p) * s * (1.0f - s);
      }
      sx[i * MLP_T + j] = x[i];
      sdz[i * MLP_T + j] = dz;
      gb2 += dz;
    }
    // an inactive unit contributes nothing even where a feature is infinite or
    // NaN: tiles with such features mask them, the others only dL/dz
    const bool mask = __syncthreads_or(!fin) != 0;
    if (!mask) {
#pragma unroll 4
      for (int i = wid; i < TILE; i += MLP_W) {
        const float4 xi = sx[i];
        const float dzi = sdz[i];
#pragma unroll
        for (int q = 0; q < MLP_UL; ++q) {
          const float pre = mlp_pre(w[q], ub[q], xi);
          const float d = pre > 0.0f ? dzi : 0.0f;
          gw2[q] = fmaf(d, fmaxf(pre, 0.0f), gw2[q]);
          gW[q].x = fmaf(d, xi.x, gW[q].x);
          gW[q].y = fmaf(d, xi.y, gW[q].y);
          gW[q].z = fmaf(d, xi.z, gW[q].z);
          gW[q].w = fmaf(d, xi.w, gW[q].w);
          gb1[q] += d;
        }
      }
    } else {
#pragma unroll 1
      for (int i = wid; i < TILE; i += MLP_W) {
        const float4 xi = sx[i];
        const float dzi = sdz[i];
#pragma unroll
        for (int q = 0; q < MLP_UL; ++q) {
          const float pre = mlp_pre(w[q], ub[q], xi);
          if (!(pre > 0.0f)) continue;
          gw2[q] = fmaf(dzi, pre, gw2[q]);
          gW[q].x = fmaf(dzi, xi.x, gW[q].x);
          gW[q].y = fmaf(dzi, xi.y, gW[q].y);
          gW[q].z = fmaf(dzi, xi.z, gW[q].z);
          gW[q].w = fmaf(dzi, xi.w, gW[q].w);
          gb1[q] += dzi;
        }
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < MLP_UL; ++q) {
    const float s[GRAD_V] = {gW[q].x, gW[q].y, gW[q].z, gW[q].w, gb1[q], gw2[q]};
#pragma unroll
    for (int f = 0; f < GRAD_V; ++f) sg[wid][f][lane + 32 * q] = s[f];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) gb2 += __shfl_xor_sync(0xffffffffu, gb2, o);
  if (lane == 0) sb[wid] = gb2;
  sl[j] = lsum;
  __syncthreads();
  // parameter-major partials: gpart[i * nb + block] (the reduction reads
  // each parameter's partials contiguously)
  const size_t nb = gridDim.x, b = blockIdx.x;
  const float w2 = su[j].w2;
#pragma unroll
  for (int f = 0; f < GRAD_V; ++f) {
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < MLP_W; ++q) s += sg[q][f][j];
    const int at = f < NF ? OFF_W1 + j * NF + f : f == NF ? OFF_B1 + j : OFF_W2 + j;
    gpart[(size_t)at * nb + b] = f <= NF ? w2 * s : s;
  }
  if (j == 0) {
    float s = 0.f;
    for (int q = 0; q < MLP_W; ++q) s += sb[q];
    gpart[(size_t)OFF_B2 * nb + b] = s;
  }
  for (int s = MLP_T / 2; s > 0; s >>= 1) {
    if (j < s) sl[j] += sl[j + s];
    __syncthreads();
  }
  if (j == 0) lpart[blockIdx.x] = sl[0];
}

// One warp per parameter (warp NPARAM: the loss): the lanes sum strided runs of
// the partials, then a fixed-order tree of shuffles, so the result is
// deterministic.  out = (accumulate ? out : 0) + weight * sum.
constexpr int RED_T = 128;
__global__ void __launch_bounds__(RED_T) k_mlp_grad_reduce(const float* __restrict__ gpart,
                                                           const double* __restrict__ lpart, int nb, double inv_n,
                                                           float weight, int accumulate, float* __restrict__ grad,
                                                           float* __restrict__ loss) {
  const int lane = threadIdx.x & 31;
  const int i = (int)(blockIdx.x * (RED_T / 32) + (threadIdx.x >> 5));
  if (i > NPARAM) return;
  double s = 0.0;
  if (i < NPARAM) {
#pragma unroll 8
    for (int b = lane; b < nb; b += 32) s += (double)gpart[(size_t)i * nb + b];
  } else {
#pragma unroll 8
    for (int b = lane; b < nb; b += 32) s += lpart[b];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane != 0) return;
  if (i < NPARAM) {
    const float v = weight * (float)s;
    grad[i] = accumulate ? grad[i] + v : v;
  } else if (loss != nullptr) {
    const float v = weight * (float)(s * inv_n);
    *loss = accumulate ? *loss + v : v;
  }
}

__global__ void k_adam(int32_t count, float* __restrict__ params, const float* __restrict__ grad,
                       float* __restrict__ m, float* __restrict__ v, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const float g = grad[i];
  const float mi = b1 * m[i] + (1.0f - b1) * g;
  const float vi = b2 * v[i] + (1.0f - b2) * g * g;
  m[i] = mi;
  v[i] = vi;
  params[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// Vertices per thread, at most `most`: two blocks per SM at least.
static int mlp_vertices(int32_t n, int most) {
  while (most > 1 && n < (int64_t)152 * 2 * most * MLP_T) most /= 2;
  return most;
}

// Blocks for n vertices in tiles of `tile`: at most eight per SM, with equal
// numbers of tiles.
static int mlp_blocks(int32_t n, int tile) {
  const int64_t tiles = ((int64_t)n + tile - 1) / tile;
  const int64_t per = (tiles + 152 * 8 - 1) / (152 * 8);
  return (int)((tiles + per - 1) / per);
}

}  // namespace fcx

using namespace fcx;

extern "C" int32_t fc_mlp_param_count(void) { return NPARAM; }

extern "C" fc_status fc_vertex_features(fc_graph* g, int32_t alpha_idx, float* X, void* stream) {
  if (g == nullptr || X == nullptr || alpha_idx < 0 || alpha_idx >= g->n_alpha) {
    set_error("fc_vertex_features: bad argument");
    return FC_EINVAL;
  }
  cudaStream_t st = (cudaStream_t)stream;
  unsigned long long* s2 = nullptr;
  FC_CK(cudaMallocAsync((void**)&s2, (size_t)g->n * sizeof(unsigned long long), st));
  FC_CK(cudaMemsetAsync(s2, 0, (size_t)g->n * sizeof(unsigned long long), st));
  const int64_t tiles = (g->nnz + NDS_TILE - 1) / NDS_TILE;
  if (tiles > 0) {
    const int64_t per = (tiles + 152 * 6 - 1) / (152 * 6);  // consecutive tiles per block, six blocks per SM
    k_nbr_deg_sum<<<(unsigned)((tiles + per - 1) / per), NDS_T, 0, st>>>(g->n, g->nnz, g->rowptr, g->colidx, g->deg,
                                                                         per, s2);
    FC_LAUNCHED();
  }
  const unsigned fb = (unsigned)std::min<int64_t>(((int64_t)g->n + 255) / 256, 152 * 16);
  k_features<<<fb, 256, 0, st>>>(g->n, g->alphas[alpha_idx], g->alpha_v, g->deg, g->dw, s2, (float4*)X);
  FC_LAUNCHED();
  FC_CK(cudaFreeAsync(s2, st));
  return FC_OK;
}

extern "C" fc_status fc_mlp_forward(fc_graph* g, int32_t alpha_idx, const float* X, const float* params,
                                    float* g_out, void* stream) {
  if (g == nullptr || X == nullptr || params == nullptr || g_out == nullptr || alpha_idx < 0 ||
      alpha_idx >= g->n_alpha) {
    set_error("fc_mlp_forward: bad argument");
    return FC_EINVAL;
  }
  cudaStream_t st = (cudaStream_t)stream;
  // vertices per thread: the most that still gives every SM two blocks, as for
  // the gradient (a thread's vertices share its loads, but run one after another)
  const int nv = mlp_vertices(g->n, 8);
  (nv == 8 ? k_mlp_forward<8> : nv == 4 ? k_mlp_forward<4> : nv == 2 ? k_mlp_forward<2> : k_mlp_forward<1>)
      <<<mlp_blocks(g->n, nv * MLP_T), MLP_T, 0, st>>>(g->n, (const float4*)X, g->rowinfo + (size_t)alpha_idx * g->n,
                                                       params, g_out);
  FC_LAUNCHED();
  return FC_OK;
}

extern "C" fc_status fc_mlp_loss_grad_acc(fc_graph* g, int32_t alpha_idx, const float* X, const float* y,
                                          const float* params, float weight, int32_t accumulate, float* grad,
                                          float* loss, void* stream) {
  if (g == nullptr || X == nullptr || y == nullptr || params == nullptr || grad == nullptr || alpha_idx < 0 ||
      alpha_idx >= g->n_alpha || !std::isfinite(weight)) {
    set_error("fc_mlp_loss_grad: bad argument");
    return FC_EINVAL;
  }
  cudaStream_t st = (cudaStream_t)stream;
  // vertices per thread: the most that still gives every SM two blocks (GB300,
  // whole calls with 1, 2, 4 vertices: n = 2^16 24, 27, - us; 2^17 37, 29, 34;
  // 2^18 54, 45, 42; 2^22 -, 425, 397)
  const int nv = mlp_vertices(g->n, 4);
  const int nb = mlp_blocks(g->n, nv * MLP_T);
  float* gpart = nullptr;
  double* lpart = nullptr;
  FC_CK(cudaMallocAsync((void**)&gpart, (size_t)nb * NPARAM * sizeof(float), st));
  FC_CK(cudaMallocAsync((void**)&lpart, (size_t)nb * sizeof(double), st));
  (nv == 4 ? k_mlp_grad<4> : nv == 2 ? k_mlp_grad<2> : k_mlp_grad<1>)<<<nb, MLP_T, 0, st>>>(
      g->n, (const float4*)X, g->rowinfo + (size_t)alpha_idx * g->n, y, params,
                                   1.0f / (float)g->n, gpart, lpart);
  FC_LAUNCHED();
  k_mlp_grad_reduce<<<(NPARAM + RED_T / 32) / (RED_T / 32), RED_T, 0, st>>>(gpart, lpart, nb, 1.0 / (double)g->n, weight, accumulate ? 1 : 0,
                                                  grad, loss);
  FC_LAUNCHED();
  FC_CK(cudaFreeAsync(gpart, st));
  FC_CK(cudaFreeAsync(lpart, st));
  return FC_OK;
}

extern "C" fc_status fc_mlp_loss_grad(fc_graph* g, int32_t alpha_idx, const float* X, const float* y,
                                      const float* params, float* grad, float* loss, void* stream) {
  return fc_mlp_loss_grad_acc(g, alpha_idx, X, y, params, 1.0f, 0, grad, loss, stream);
}

extern "C" fc_status fc_mlp_adam(float* params, const float* grad, float* m, float* v, int32_t count, int32_t step,
                                 float lr, float beta1, float beta2, float eps, void* stream) {
  if (params == nullptr || grad == nullptr || m == nullptr || v == nullptr || count < 1 || step < 1) {
    set_error("fc_mlp_adam: bad argument");
    return FC_EINVAL;
  }
  cudaStream_t st = (cudaStream_t)stream;
  const float c1 = 1.0f - powf(beta1, (float)step);
  const float c2 = 1.0f - powf(beta2, (float)step);
  k_adam<<<(count + 255) / 256, 256, 0, st>>>(count, params, grad, m, v, lr, beta1, beta2, eps, c1, c2);
  FC_LAUNCHED();
  return FC_OK;
}
