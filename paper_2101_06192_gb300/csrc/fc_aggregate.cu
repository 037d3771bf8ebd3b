// Tree-path aggregation over sampled trees: forest roots and depths, and
// root-frequency counts.
//
// In a spanning tree of G* rooted at u*, removing u* leaves a rooted spanning
// forest of G whose roots are the children of u*.  By the matrix-forest
// theorem (Sec. 2), Omega[u, v] is the probability that v's tree of that
// forest is rooted at u, so root frequencies over sampled trees estimate whole
// columns of Omega (the diagonal is Prop. 1's u*-edge frequency), and with them
// pairwise forest distances rho(u, v) = Omega_uu + Omega_vv - 2 Omega_uv
// (Def. 1).
//
// fc_tree_roots: pointer jumping, one cooperative launch.  Every node walks
// AG_HOPS0 steps over the parents and keeps a 64-bit word {ancestor, distance to
// it, done}, done when the ancestor is a root (parent u*).  A round replaces
// each word that is not done by {ancestor of its ancestor, summed distance, done
// of the ancestor}, AG_HOPS times, so O(log depth) rounds end with every node at
// its root and depth; a done node reads only its own word.  Words are read and
// written whole, so a node may read a word of this round or the last one.  A
// parent cycle never reaches a root and is caught by the round limit.  The trees
// are taken in windows of AG_WINDOW bytes of words, which bounds the workspace.
// Bound by the gathers of parents and words, four in flight per thread: on
// GB300, BA n = 2^20, 152 trees, with the copies of the status, 10.5 -> 4.4 ms
// against a launch per round over all trees with a host read between rounds that
// gathered for done nodes too; windows of 64 MB 4.4, all trees at once 4.8, with
// one jump per round 11.3 (8 MB) to 4.8 (all at once); 0.45 -> 0.40 ms for BA
// n = 2^17, 96 trees from one jump per round to two.
// (A first version took one CTA per tree with children lists and BFS levels;
// its per-tree scratch, touched at random, moved 60x the algorithmic bytes.)
#include <cooperative_groups.h>

#include <algorithm>

#include "fc_internal.cuh"

namespace fcx {

constexpr int AG_T = 256;
constexpr int AG_U = 4;                      // nodes per thread and task: loads in flight
constexpr int AG_CHUNK = AG_U * AG_T;        // vertices of one tree per task
constexpr int AG_HOPS0 = 4;                  // steps over the parents before the first round
constexpr int AG_HOPS = 2;                   // jumps per round
constexpr int AG_ROUNDS = 34;                // depth < n < 2^31 needs at most 32
constexpr int64_t AG_WINDOW = 64ll << 20;    // bytes of words of a window (at least one tree)
constexpr unsigned long long AG_DONE = 1ull << 63;

__device__ __forceinline__ unsigned long long rw_pack(int32_t a, uint32_t d, bool done) {
  return (unsigned long long)(uint32_t)a | ((unsigned long long)(d & 0x7fffffffu) << 32) | (done ? AG_DONE : 0ull);
}
__device__ __forceinline__ unsigned long long rw_load(const unsigned long long* p) {
  unsigned long long w;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
  return w;
}
__device__ __forceinline__ void rw_store(unsigned long long* p, unsigned long long w) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}

// The T trees in windows of wt; jw: the words of one window.  parents may be
// roots or depth (a window's parents are read before its first barrier, its
// roots written after).  state: [0] error, [1..3] nodes not done, by round mod
// 3 (zeroed)
__global__ void __launch_bounds__(AG_T) k_roots(const int32_t* parents, int32_t n, int64_t T, int64_t wt,
                                                unsigned long long* jw, int32_t* roots, int32_t* depth,
                                                uint32_t* __restrict__ state) {
  cooperative_groups::grid_group grid = cooperative_groups::this_grid();
  const int64_t chunks = ((int64_t)n + AG_CHUNK - 1) / AG_CHUNK;
  int slot = 1;
  for (int64_t t0 = 0; t0 < T; t0 += wt) {
    const int64_t tasks = (T - t0 < wt ? T - t0 : wt) * chunks;
    // f(index of the tree's vertex 0 in the window, first vertex of the thread) over this block's tasks
    auto each = [&](auto f) {
      for (int64_t task = blockIdx.x; task < tasks; task += gridDim.x) {
        const int64_t t = task / chunks;
        f(t * n, (uint32_t)(task - t * chunks) * AG_CHUNK + threadIdx.x);
      }
    };
    const int64_t off = t0 * n;
    bool bad = false;
    // the words of a thread's own nodes: no barrier after the window before
    each([&](int64_t base, uint32_t v0) {
      const int32_t* par = parents + off + base;
      int32_t a[AG_U], q[AG_U];
      uint32_t d[AG_U];
      bool live[AG_U], done[AG_U];
#pragma unroll
      for (int i = 0; i < AG_U; ++i) {
        a[i] = (int32_t)(v0 + i * AG_T);
        d[i] = 0u;
        live[i] = v0 + i * AG_T < (uint32_t)n;
        done[i] = false;
      }
#pragma unroll
      for (int h = 0; h < AG_HOPS0; ++h) {
#pragma unroll
        for (int i = 0; i < AG_U; ++i) q[i] = live[i] ? par[a[i]] : 0;
#pragma unroll
        for (int i = 0; i < AG_U; ++i) {
          if (!live[i]) continue;
          done[i] = q[i] == n;
          const bool wrong = q[i] < 0 || q[i] > n || q[i] == a[i];
          bad |= wrong;
          live[i] = !done[i] && !wrong;
          if (live[i]) {
            a[i] = q[i];
            ++d[i];
          }
        }
      }
#pragma unroll
      for (int i = 0; i < AG_U; ++i)
        if (v0 + i * AG_T < (uint32_t)n) rw_store(jw + base + v0 + i * AG_T, rw_pack(a[i], d[i], done[i]));
    });
    if (bad) atomicOr(&state[0], ERR_INVAL);
    grid.sync();
    if (*(volatile uint32_t*)&state[0] != 0u) return;  // uniform: written before the barrier
    for (int r = 0;; ++r) {
      const int next = slot == 3 ? 1 : slot + 1;
      bool open = false;
      each([&](int64_t base, uint32_t v0) {
        unsigned long long w[AG_U], x[AG_U];
        bool go[AG_U];
#pragma unroll
        for (int i = 0; i < AG_U; ++i)
          w[i] = v0 + i * AG_T < (uint32_t)n ? rw_load(jw + base + v0 + i * AG_T) : AG_DONE;
#pragma unroll
        for (int i = 0; i < AG_U; ++i) go[i] = (w[i] & AG_DONE) == 0ull;
#pragma unroll
        for (int k = 0; k < AG_HOPS; ++k) {
#pragma unroll
          for (int i = 0; i < AG_U; ++i)
            if ((w[i] & AG_DONE) == 0ull) x[i] = rw_load(jw + base + (uint32_t)w[i]);
#pragma unroll
          for (int i = 0; i < AG_U; ++i)
            if ((w[i] & AG_DONE) == 0ull)
              w[i] = rw_pack((int32_t)(uint32_t)x[i], (uint32_t)(w[i] >> 32) + ((uint32_t)(x[i] >> 32) & 0x7fffffffu),
                             (x[i] & AG_DONE) != 0ull);
        }
#pragma unroll
        for (int i = 0; i < AG_U; ++i) {
          if (go[i]) rw_store(jw + base + v0 + i * AG_T, w[i]);
          open |= (w[i] & AG_DONE) == 0ull;
        }
      });
      if (__syncthreads_or(open) && threadIdx.x == 0) atomicOr(&state[slot], 1u);
      if (blockIdx.x == 0 && threadIdx.x == 0) state[next] = 0u;  // read two rounds ago
      grid.sync();
      const bool more = *(volatile uint32_t*)&state[slot] != 0u;  // uniform
      slot = next;
      if (!more) break;
      if (r == AG_ROUNDS) {  // a parent cycle
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&state[0], ERR_INVAL);
        return;
      }
    }
    each([&](int64_t base, uint32_t v0) {
#pragma unroll
      for (int i = 0; i < AG_U; ++i) {
        const uint32_t v = v0 + i * AG_T;
        if (v >= (uint32_t)n) continue;
        const unsigned long long w = jw[base + v];
        if (roots) roots[off + base + v] = (int32_t)(uint32_t)w;
        if (depth) depth[off + base + v] = (int32_t)((w >> 32) & 0x7fffffffull);
      }
    });
  }
}

// counts[q][v] += #{t : roots[t][v] == queries[q]}; qidx[u] = q or -1
__global__ void k_root_counts(const int32_t* __restrict__ roots, int32_t n, int64_t T,
                              const int32_t* __restrict__ qidx, uint32_t* __restrict__ counts) {
  const size_t total = (size_t)T * (size_t)n;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const int32_t r = roots[i];
    if (r < 0 || r >= n) continue;
    const int32_t q = qidx[r];
    if (q >= 0) atomicAdd(&counts[(size_t)q * n + (i % (size_t)n)], 1u);
  }
}

__global__ void k_qidx(int32_t n, const int32_t* __restrict__ queries, int32_t k, int32_t* __restrict__ qidx,
                       uint32_t* err) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < k) {
    const int32_t u = queries[i];
    if (u < 0 || u >= n) atomicOr(err, ERR_INVAL);
    else atomicCAS(&qidx[u], -1, i);  // first query wins for duplicates
  }
}

fc_status tree_roots(const int32_t* parents, int32_t n, int64_t T, int32_t* roots, int32_t* depth, cudaStream_t st) {
  int nsm = 0, dev = 0;
  FC_CK(cudaGetDevice(&dev));
  FC_CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  int coop = 0, per_sm = 0;
  FC_CK(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
  FC_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_roots, AG_T, 0));
  if (!coop || per_sm < 1) {
    set_error("fc_tree_roots: the device does not support cooperative launches");
    return FC_ECUDA;
  }
  const int64_t wt = std::min(T, std::max<int64_t>(1, AG_WINDOW / ((int64_t)n * 8)));
  const int64_t N = wt * (int64_t)n, tasks = wt * (((int64_t)n + AG_CHUNK - 1) / AG_CHUNK);
  const unsigned blocks = (unsigned)std::min<int64_t>(tasks, (int64_t)nsm * per_sm);
  unsigned long long* jw = nullptr;
  uint32_t* state = nullptr;
  FC_CK(cudaMallocAsync((void**)&jw, (size_t)N * sizeof(unsigned long long) + 16, st));
  state = (uint32_t*)(jw + N);
  FC_CK(cudaMemsetAsync(state, 0, 16, st));
  void* args[] = {&parents, &n, &T, (void*)&wt, &jw, &roots, &depth, &state};
  FC_CK(cudaLaunchCooperativeKernel((const void*)k_roots, dim3(blocks), dim3(AG_T), args, 0, st));
  FC_LAUNCHED();
  uint32_t h = 0;
  FC_CK(cudaMemcpyAsync(&h, state, sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
  FC_CK(cudaFreeAsync(jw, st));
  FC_CK(cudaStreamSynchronize(st));
  if (h != 0u) {
    set_error("fc_tree_roots: parents do not form spanning trees rooted at u* = n");
    return FC_EINVAL;
  }
  return FC_OK;
}

}  // namespace fcx

using namespace fcx;

extern "C" fc_status fc_tree_roots(const int32_t* parents, int32_t n, int64_t T, int32_t* roots, int32_t* depth,
                                   void* stream) {
  if (parents == nullptr || roots == nullptr || n < 1 || T < 0) {
    set_error("fc_tree_roots: bad argument");
    return FC_EINVAL;
  }
  if (T == 0) return FC_OK;
  return tree_roots(parents, n, T, roots, depth, (cudaStream_t)stream);
}

extern "C" fc_status fc_root_counts(const int32_t* roots, int32_t n, int64_t T, const int32_t* queries, int32_t k,
                                    uint32_t* counts, void* stream) {
  if (roots == nullptr || queries == nullptr || counts == nullptr || n < 1 || T < 0 || k < 1) {
    set_error("fc_root_counts: bad argument");
    return FC_EINVAL;
  }
  cudaStream_t st = (cudaStream_t)stream;
  int32_t* qidx = nullptr;
  uint32_t* err = nullptr;
  FC_CK(cudaMallocAsync((void**)&qidx, (size_t)n * sizeof(int32_t), st));
  FC_CK(cudaMallocAsync((void**)&err, sizeof(uint32_t), st));
  FC_CK(cudaMemsetAsync(qidx, 0xff, (size_t)n * sizeof(int32_t), st));
  FC_CK(cudaMemsetAsync(err, 0, sizeof(uint32_t), st));
  k_qidx<<<(k + 255) / 256, 256, 0, st>>>(n, queries, k, qidx, err);
  FC_LAUNCHED();
  if (T > 0) {
    const size_t total = (size_t)T * (size_t)n;
    const unsigned blocks = (unsigned)std::min<size_t>((total + 255) / 256, 152 * 64);
    k_root_counts<<<blocks, 256, 0, st>>>(roots, n, T, qidx, counts);
    FC_LAUNCHED();
  }
  uint32_t herr = 0;
  FC_CK(cudaMemcpyAsync(&herr, err, sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
  FC_CK(cudaFreeAsync(qidx, st));
  FC_CK(cudaFreeAsync(err, st));
  FC_CK(cudaStreamSynchronize(st));
  if (herr) {
    set_error("fc_root_counts: query vertex out of range");
    return FC_EINVAL;
  }
  return FC_OK;
}
