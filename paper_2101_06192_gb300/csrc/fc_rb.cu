// Rao-Blackwellised estimate of diag(Omega) from sampled trees: an estimator
// on the same samples as Prop. 1 (not in the paper).
//
// With the parents of all vertices but v fixed, the vertices whose path to
// u* runs through v (v's subtree S(v), v included) are fixed, and v's parent
// can be u* (edge weight 1) or any neighbour w outside S(v) (edge weight
// alpha w_vw); every choice gives a spanning tree of G* whose weight is the
// same product times that edge's weight.  So
//     P(parent(v) = u* | the other parents) = 1 / (1 + alpha sum_{w in N(v)\S(v)} w_vw),
// and its average over trees is unbiased for Omega[v, v] with at most the
// variance of the indicator.  w in S(v) iff tin[v] <= tin[w] < tin[v] +
// size[v] for a preorder numbering tin and subtree sizes.  The sum runs over
// v's CSR row in order in FP64 and the value 1 / (1 + alpha s) is rounded
// once per operation; per tree it is added in fixed point, floor(value *
// 2^48 + 1/2), so totals do not depend on the order of the additions.
//
// One cooperative kernel handles a chunk of up to 32 trees with every
// resident CTA; grid-wide barriers separate the phases, and none of them
// takes a barrier per tree level, so deep trees cost no more barriers than
// shallow ones: child counts (with validation); subtree sizes and sibling
// offsets by peeling leaves (one atomic per tree node, the node finished by
// whichever thread delivers its last child); the roots' offsets; preorder
// numbers by pointer jumping down the paths (O(log depth) rounds); and the rows
// with the per-vertex sums.  Preorder numbers and sizes are stored vertex-major
// across the chunk's trees, so a warp scanning a row with one lane per tree
// reads each neighbour's numbers for all trees in one 128-byte line.  Long
// unweighted rows are split into segments of 256 entries whose counts add
// up exactly; a weighted row stays with one warp so that each lane adds its
// tree's weights in row order.  Every loop bound and every early exit is
// read from global memory after a barrier, so all CTAs take the same path
// through the barriers.
//
// Bound by latency: the atomic chains of the peeling and the neighbours' lines.
// Measured on GB300, 32 trees of R-MAT n = 2^18, m = 16: whole call 1470 ->
// 1160 us.  Phases (with a clock read at each barrier): counts 52 -> 35;
// peeling 410 -> 265 (children and sizes in one word, sizes read from it in the
// end, idle lanes fed from a ring instead of by searching bit masks); roots'
// offsets 165 -> 45 (a block scan and an atomic per 1024 vertices instead of a
// grid-wide scan of all nodes); jumping 220 -> 175 (four loads in flight, two
// jumps per round); rows about 470 -> 440 (no loads for leaves, one-segment rows
// finished at once).  Four CTAs per SM: with five, registers spill (1300 us);
// 16 loads in flight or rows from a shared counter change nothing (1160, 1150).
//
// The same kernel, in its second mode, aggregates the effective resistances
// r(u, v) between a pivot u and every vertex v (Sec. 3, insight (iii)) from
// uniform spanning trees of G rooted at u (sampled on a graph from
// fc_build_rooted, whose trees are u* -> u -> ...).  Kirchhoff's current
// theorem: a unit current from v to u puts current P(a->b) - P(b->a) on an
// edge {a, b}, where P(a->b) is the probability that v's tree path to u
// crosses it from a to b; summing current / w along any fixed path from v to
// u (here v's path in a breadth-first tree B of u) gives r(u, v).  Per tree,
//   S_T(v) = sum over the edges (x, b(x)) of v's B-path, from v upward, of
//            ( [par_T(x) = b(x), x ancestor-or-self of v in T]
//            - [par_T(b(x)) = x, b(x) ancestor-or-self of v in T] ) / w(x, b(x)),
// summed in FP64 in path order and added in signed fixed point
// floor(S_T(v) 2^32 + 1/2).  Ancestry uses the same preorder numbers and
// subtree sizes; a warp takes a vertex and walks its B-path once for the
// chunk's trees (one lane per tree, tree parents stored vertex-major).
#include <cooperative_groups.h>

#include <algorithm>

#include "fc_internal.cuh"

namespace cg = cooperative_groups;

namespace fcx {

namespace {

constexpr int RB_T = 256;
constexpr int RB_FRAC = 48;
constexpr int RB_SEG = 256;  // entries per segment of a long unweighted row
constexpr int RB_TMAX = 32;  // trees per chunk: one per lane of a warp

struct RBParams {
  int32_t n;
  int32_t Tc;                 // trees in this chunk (at most 32: one per lane)
  const int64_t* rowptr;
  const int32_t* colidx;
  const float* w;             // or null
  double alpha;
  const double* alpha_v;      // per-vertex alpha (batches) or null
  const int32_t* parents;     // [Tc][n]
  uint64_t* acc;              // [n] fixed-point sums
  const int4* segs;           // row segments {v, entries, first entry (low, high word)}
  const uint32_t* nseg;       // number of segments
  // scratch.  Per tree node flat index i = t n + v; vertex-major index v Tc + t.
  unsigned long long* word;   // [Tc n] {children not finished, summed sizes of the finished ones} (zeroed)
  unsigned long long* jw;     // [Tc n] pointer-jumping words {ancestor, partial preorder number}
  int32_t* size;              // [n][Tc] subtree sizes (vertex-major)
  int32_t* tin;               // [n][Tc] preorder numbers (vertex-major)
  uint32_t* outc;             // [n][Tc] rows of several segments: count of neighbours outside the subtree
  uint32_t* tsum;             // [Tc] vertices below the tree's roots so far (zeroed)
  uint32_t* ctr;              // [2] error, [4..6] open flags of the jumping rounds, [7] chunk grabs (zeroed)
  const uint64_t* qtab;       // unweighted, one alpha: fixed-point value for each count of outside neighbours, or null
  // resistance mode
  int32_t root;               // the pivot u (the only child of u*), -1 in the diag(Omega) mode
  const int32_t* bpar;        // [n] breadth-first parent of each vertex (-1 at the root)
  const double* binv;         // [n] 1 / w(v, bpar(v))
  int64_t* racc;              // [n] signed fixed-point totals of S_T(v)
  int32_t* pvm;               // [n][Tc] tree parents, vertex-major
};

constexpr int RES_FRAC = 32;

__device__ __forceinline__ uint32_t block_exscan_u32(uint32_t x, uint32_t* total, uint32_t* wsum) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t s = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
    if (lane >= o) s += y;
  }
  if (lane == 31) wsum[wid] = s;
  __syncthreads();
  if (wid == 0) {
    uint32_t t = lane < (int)(blockDim.x >> 5) ? wsum[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    wsum[lane] = t;
  }
  __syncthreads();
  const uint32_t ex = s - x + (wid > 0 ? wsum[wid - 1] : 0u);
  *total = wsum[(blockDim.x >> 5) - 1];
  __syncthreads();
  return ex;
}

__device__ __forceinline__ unsigned long long jw_pack(int32_t anc, int32_t sum) {
  return (unsigned long long)(uint32_t)anc | ((unsigned long long)(uint32_t)sum << 32);
}

constexpr int RB_TILE = RB_T;  // vertices per tile of the vertex-major transpose

__device__ __forceinline__ unsigned long long jw_load(const unsigned long long* p) {
  unsigned long long w;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
  return w;
}
__device__ __forceinline__ void jw_store(unsigned long long* p, unsigned long long w) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}

constexpr int RB_U = 4;               // nodes per thread and task: loads in flight
constexpr int RB_CHUNK = RB_U * RB_T; // vertices of one tree per task
constexpr int RB_RING = 64;           // leaves of a warp waiting for a lane

// MODE 0: Rao-Blackwellised diag(Omega); MODE 1: effective resistances to the pivot.
template <int MODE>
__global__ void __launch_bounds__(RB_T, 4) k_rb(RBParams p) {
  cg::grid_group grid = cg::this_grid();
  __shared__ int32_t tile[RB_TMAX][RB_TILE + 1];
  __shared__ uint32_t wsum[32];
  __shared__ uint32_t sbase;
  const int32_t n = p.n;
  const int32_t Tc = p.Tc;
  const int64_t N = (int64_t)Tc * n;  // below 2^31
  const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t gstride = (int64_t)gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31;
  const int64_t gwarp = gtid >> 5, nwarps = gstride >> 5;
#define VT(t, v) ((int64_t)(v) * Tc + (t))
  const int32_t chunks = (int32_t)(((int64_t)n + RB_CHUNK - 1) / RB_CHUNK);
  // f(tree, flat index of its vertex 0, first vertex of the block) over this block's tasks
  auto each = [&](auto f) {
    for (int32_t task = blockIdx.x; task < Tc * chunks; task += gridDim.x) {
      const int32_t t = task / chunks;
      f(t, (int64_t)t * n, (uint32_t)(task - t * chunks) * RB_CHUNK);
    }
  };

  // ---- child counts; parents must lie in [0, n] and differ from the vertex ----
  each([&](int32_t t, int64_t b, uint32_t c0) {
#pragma unroll
    for (int i = 0; i < RB_U; ++i) {
      const uint32_t v = c0 + i * RB_T + threadIdx.x;
      if (v >= (uint32_t)n) continue;
      const int32_t par = p.parents[b + v];
      if (par < 0 || par > n || par == (int32_t)v) atomicOr(&p.ctr[2], ERR_INVAL);
      // a tree of G rooted at the pivot: the pivot, and only the pivot, hangs from u*
      else if (MODE == 1 && ((par == n) != ((int32_t)v == p.root))) atomicOr(&p.ctr[2], ERR_INVAL);
      else if (par < n) atomicAdd(&p.word[b + par], 1ull << 32);  // u*'s children: a scan below
    }
  });
  grid.sync();
  if (*(volatile uint32_t*)&p.ctr[2] != 0u) return;  // uniform: read after the barrier

  // ---- subtree sizes and sibling offsets by peeling leaves.  A finished
  // child adds {-1, its size} to its parent's word in one atomic; the sizes
  // already there are its earlier-finished siblings', so 1 + that sum is its
  // offset in the parent's preorder interval (any sibling order gives valid
  // intervals, and subtree membership does not depend on it), and a node's
  // size is 1 + the sum of its word in the end.  The thread that delivers a
  // parent's last child carries on with the parent: no barrier per tree level.
  // The roots (u*'s children, often most vertices) take their offsets below
  // instead of from one contended word.  Warps take candidates in chunks of 32
  // (coalesced, one chunk ahead) from a shared counter, eight chunks per grab,
  // and put the leaves among them into a ring from which idle lanes take.  The
  // last deliverer of a node carries on with it, so chains pile up on some
  // lanes; warps so held up take fewer chunks.  A step loads the grandparent
  // before its atomic, so both are in flight together. ----
  {
    const unsigned lt = (1u << lane) - 1u;
    const int64_t nchunks = (N + 31) / 32;
    int32_t* ring_v = &tile[0][0] + (threadIdx.x >> 5) * 3 * RB_RING;  // vertex, parent, flat index of the tree's vertex 0
    int32_t* ring_p = ring_v + RB_RING;
    int32_t* ring_b = ring_p + RB_RING;
    unsigned head = 0, cnt = 0;  // warp-uniform
    int64_t sc = 0;              // current grab (warp-uniform)
    int kc = 8;                  // next chunk within it
    bool dry = false;
    int32_t nb = 0, nv = 0, np = n;  // prefetched chunk: this lane's node
    bool nleaf = false;
    bool pre = false;  // a prefetched chunk is waiting (warp-uniform)
    auto load = [&]() {
      pre = false;
      nleaf = false;
      if (dry) return;
      if (kc == 8) {
        uint32_t g = 0;
        if (lane == 0) g = atomicAdd(&p.ctr[7], 1u);
        sc = __shfl_sync(0xffffffffu, g, 0);
        kc = 0;
      }
      const int64_t c = sc * 8 + kc++;
      if (c >= nchunks) {
        dry = true;
        return;
      }
      pre = true;
      const uint32_t i = (uint32_t)(c * 32) + lane;
      if (i < (uint32_t)N) {
        np = p.parents[i];
        // (the word of a node whose children are all finished holds their sizes)
        nleaf = *(volatile unsigned long long*)&p.word[i] == 0ull && np != n;
        const uint32_t t = i / (uint32_t)n;
        nb = (int32_t)(t * (uint32_t)n);
        nv = (int32_t)i - nb;
      }
    };
    load();
    int32_t b = 0, v = -1, par = 0;  // this lane's node (none: v < 0)
    uint32_t s = 0;
    for (;;) {
      while (pre && cnt < 32u) {
        const unsigned lm = __ballot_sync(0xffffffffu, nleaf);
        if (nleaf) {
          const unsigned at = (head + cnt + __popc(lm & lt)) & (RB_RING - 1);
          ring_v[at] = nv;
          ring_p[at] = np;
          ring_b[at] = nb;
        }
        cnt += __popc(lm);
        load();
      }
      __syncwarp();
      const unsigned need = __ballot_sync(0xffffffffu, v < 0);
      if (need == 0xffffffffu && cnt == 0u) break;  // uniform (nothing prefetched: the loop above drained it)
      const unsigned r = __popc(need & lt);
      if (v < 0 && r < cnt) {
        const unsigned at = (head + r) & (RB_RING - 1);
        v = ring_v[at];
        par = ring_p[at];
        b = ring_b[at];
        s = 1u;
      }
      const unsigned took = min((unsigned)__popc(need), cnt);
      head += took;
      cnt -= took;
      __syncwarp();
      if (v < 0) continue;
      const int32_t pi = b + par;
      const int32_t gp = p.parents[pi];
      const unsigned long long old = atomicAdd(&p.word[pi], (0xffffffffull << 32) | s);
      p.jw[b + v] = jw_pack(pi, (int32_t)(1u + (uint32_t)old));
      if ((uint32_t)(old >> 32) != 1u || gp == n) {
        v = -1;
        continue;
      }
      s = 1u + (uint32_t)old + s;
      v = par;
      par = gp;
    }
  }
  grid.sync();
  // roots: preorder number = sizes of the tree's roots before it, by chunk in
  // the order in which the blocks add up (any order of the roots will do)
  each([&](int32_t t, int64_t b, uint32_t c0) {
    uint32_t x[RB_U], s = 0;
    bool root[RB_U];
#pragma unroll
    for (int i = 0; i < RB_U; ++i) {
      const uint32_t v = c0 + i * RB_T + threadIdx.x;
      root[i] = v < (uint32_t)n && p.parents[b + v] == n;
      const unsigned long long w = root[i] ? *(volatile unsigned long long*)&p.word[b + v] : 0ull;
      x[i] = s;
      // (children left: the root of an unfinished tree, never in a forest)
      s += root[i] && (w >> 32) == 0ull ? 1u + (uint32_t)w : 0u;
    }
    uint32_t tot = 0;
    const uint32_t ex = block_exscan_u32(s, &tot, wsum);
    if (threadIdx.x == 0) sbase = tot ? atomicAdd(&p.tsum[t], tot) : 0u;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < RB_U; ++i)
      if (root[i]) p.jw[b + c0 + i * RB_T + threadIdx.x] = jw_pack(-1, (int32_t)(sbase + ex + x[i]));
    __syncthreads();
  });
  grid.sync();
  // a parent cycle leaves its vertices and their subtrees outside u*'s tree
  if (__syncthreads_or(threadIdx.x < Tc && *(volatile uint32_t*)&p.tsum[threadIdx.x] != (uint32_t)n)) {
    if (gtid == 0) atomicOr(&p.ctr[2], ERR_INVAL);
    return;  // uniform: every block reads the same sums
  }

  // ---- preorder numbers: each node's number is its parent's plus its
  // offset, summed down the path by pointer jumping, two jumps per round.
  // Invariant: tin(i) = sum(i) + tin(anc(i)), with anc = -1 once sum is the
  // number itself; words are read and written whole, so a node may read an
  // ancestor's word of this round or the last one.  O(log depth) rounds. ----
  for (int r = 0;; ++r) {
    bool open = false;
    each([&](int32_t t, int64_t b, uint32_t c0) {
      unsigned long long w[RB_U], x[RB_U];
      bool go[RB_U];
#pragma unroll
      for (int i = 0; i < RB_U; ++i) {
        const uint32_t v = c0 + i * RB_T + threadIdx.x;
        w[i] = v < (uint32_t)n ? jw_load(p.jw + b + v) : jw_pack(-1, 0);
      }
#pragma unroll
      for (int i = 0; i < RB_U; ++i) go[i] = (int32_t)(uint32_t)w[i] >= 0;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int i = 0; i < RB_U; ++i)
          if ((int32_t)(uint32_t)w[i] >= 0) x[i] = jw_load(p.jw + (uint32_t)w[i]);
#pragma unroll
        for (int i = 0; i < RB_U; ++i)
          if ((int32_t)(uint32_t)w[i] >= 0)
            w[i] = jw_pack((int32_t)(uint32_t)x[i], (int32_t)((uint32_t)(w[i] >> 32) + (uint32_t)(x[i] >> 32)));
      }
#pragma unroll
      for (int i = 0; i < RB_U; ++i) {
        if (go[i]) jw_store(p.jw + b + c0 + i * RB_T + threadIdx.x, w[i]);
        open |= (int32_t)(uint32_t)w[i] >= 0;
      }
    });
    if (__syncthreads_or(open) && threadIdx.x == 0) atomicOr(&p.ctr[4 + r % 3], 1u);
    if (gtid == 0) p.ctr[4 + (r + 1) % 3] = 0u;  // read two rounds ago, after that round's barrier
    grid.sync();
    if (*(volatile uint32_t*)&p.ctr[4 + r % 3] == 0u) break;  // uniform
    if (r >= 64) {  // depth below 2^31 needs at most 32 rounds
      if (gtid == 0) atomicOr(&p.ctr[2], ERR_INVAL);
      return;
    }
  }
  // preorder numbers and sizes to vertex-major order through a shared-memory
  // tile (coalesced on both sides); the counts of rows of several segments start
  // at zero
  for (int64_t v0 = (int64_t)blockIdx.x * RB_TILE; v0 < n; v0 += (int64_t)gridDim.x * RB_TILE) {
    const int32_t nv = (int32_t)std::min<int64_t>(RB_TILE, n - v0);
    const int wid = threadIdx.x >> 5;
    // tile -> [v][t]: a lane per tree, a warp per vertex
    auto flip = [&](int32_t* dst) {
      __syncthreads();
      if (lane < Tc)
        for (int x = wid; x < nv; x += RB_T / 32) dst[VT(lane, v0 + x)] = tile[lane][x];
      __syncthreads();
    };
    for (int t = 0; t < Tc; ++t)
      for (int x = threadIdx.x; x < nv; x += blockDim.x) tile[t][x] = (int32_t)(p.jw[(int64_t)t * n + v0 + x] >> 32);
    flip(p.tin);
    for (int t = 0; t < Tc; ++t)
      for (int x = threadIdx.x; x < nv; x += blockDim.x)
        tile[t][x] = (int32_t)(1u + (uint32_t)p.word[(int64_t)t * n + v0 + x]);
    flip(p.size);
    if (MODE == 0 && !p.w) {
      const int32_t x = threadIdx.x;  // RB_TILE threads
      if (x < nv && p.rowptr[v0 + x + 1] - p.rowptr[v0 + x] > RB_SEG)
        for (int t = 0; t < Tc; ++t) p.outc[VT(t, v0 + x)] = 0u;
    }
    if (MODE == 1) {  // the tree parents, vertex-major, through the same tile
      for (int t = 0; t < Tc; ++t)
        for (int x = threadIdx.x; x < nv; x += blockDim.x) tile[t][x] = p.parents[(int64_t)t * n + v0 + x];
      flip(p.pvm);
    }
  }
  grid.sync();

  if (MODE == 1) {
    // ---- path sums along the breadth-first tree: a warp per vertex, a lane
    // per tree; the B-path is the same for every lane ----
    const int32_t root = p.root;
    for (int64_t v = gwarp; v < n; v += nwarps) {
      const bool on = lane < Tc;
      const int32_t tv = on ? p.tin[VT(lane, v)] : 0;
      double s = 0.0;
      int32_t x = (int32_t)v;
      int32_t px = on ? p.pvm[VT(lane, x)] : -1;  // parent of x in this lane's tree
      int32_t hops = 0;
      while (x != root) {
        const int32_t b = __ldg(p.bpar + x);
        const double wi = __ldg(p.binv + x);
        if (b < 0 || ++hops > n) {  // not a breadth-first tree of the root: never for fc_build_rooted graphs
          atomicOr(&p.ctr[2], ERR_INVAL);
          break;
        }
        const int32_t pb = (on && b != root) ? p.pvm[VT(lane, b)] : -1;  // parent of b
        if (on) {
          int c = 0;
          if (px == b) {  // the tree crosses x -> b: on v's tree path iff x is an ancestor-or-self of v
            const int32_t t0 = p.tin[VT(lane, x)];
            if (t0 <= tv && tv < t0 + p.size[VT(lane, x)]) c = 1;
          } else if (pb == x) {  // the tree crosses b -> x
            const int32_t t0 = p.tin[VT(lane, b)];
            if (t0 <= tv && tv < t0 + p.size[VT(lane, b)]) c = -1;
          }
          if (c != 0) s = __dadd_rn(s, c > 0 ? wi : -wi);
        }
        x = b;
        px = pb;
      }
      long long q = 0;
      if (on) q = (long long)floor(__dadd_rn(__dmul_rn(s, (double)(1ull << RES_FRAC)), 0.5));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
      if (lane == 0 && q != 0) atomicAdd((unsigned long long*)&p.racc[v], (unsigned long long)q);
    }
    return;
  }

  // ---- neighbours outside the subtree: a warp per row segment, a lane per
  // tree (each lane sums its tree's weights in row order).  A lane whose tree
  // has v as a leaf loads nothing: every neighbour is outside.  A row of one
  // segment ends with its conditional probabilities, summed over the trees;
  // longer unweighted rows leave counts, which add up exactly.  The next
  // segment's numbers and entries are loaded while the current one is scanned. ----
  const bool on = lane < Tc;
  auto finish = [&](int32_t v, double s, uint32_t c) {  // 1 / (1 + alpha s), fixed point, to acc
    uint64_t q = 0;
    if (on && p.qtab) {
      q = p.qtab[c];  // the same FP64 steps, done once per count
    } else if (on) {
      const double a = p.alpha_v ? p.alpha_v[v] : p.alpha;
      const double val = __ddiv_rn(1.0, __dadd_rn(1.0, __dmul_rn(a, p.w ? s : (double)c)));
      q = (uint64_t)__dadd_rn(__dmul_rn(val, (double)(1ull << RB_FRAC)), 0.5);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    if (lane == 0) atomicAdd((unsigned long long*)&p.acc[v], (unsigned long long)q);
  };
  {
    const int64_t nseg = *p.nseg;
    const int4 none = make_int4(0, 0, 0, 0);
    int4 rec = gwarp < nseg ? p.segs[gwarp] : none;                     // next segment
    int4 rec2 = gwarp + nwarps < nseg ? p.segs[gwarp + nwarps] : none;  // and the one after it
    int32_t nlo = 0, nsz = 1, nu = 0;
    float nw = 0.f;
    auto prefetch = [&]() {  // the numbers and the first 32 entries of rec's row
      if (on && rec.y > 0) {
        nlo = p.tin[VT(lane, rec.x)];
        nsz = p.size[VT(lane, rec.x)];
      }
      const int64_t e0 = (int64_t)(((uint64_t)(uint32_t)rec.w << 32) | (uint32_t)rec.z);
      if (lane < rec.y) {
        nu = __ldg(p.colidx + e0 + lane);
        if (p.w) nw = __ldg(p.w + e0 + lane);
      }
    };
    prefetch();
    for (int64_t sg = gwarp; sg < nseg; sg += nwarps) {
      const int4 sv = rec;
      const int32_t lo = nlo, hi = nlo + nsz;
      const bool look = on && nsz > 1;
      int32_t uj = nu;
      float wj = nw;
      rec = rec2;
      rec2 = sg + 2 * nwarps < nseg ? p.segs[sg + 2 * nwarps] : none;
      prefetch();
      const int32_t v = sv.x;
      const int64_t e0 = (int64_t)(((uint64_t)(uint32_t)sv.w << 32) | (uint32_t)sv.z);
      double s = 0.0;
      uint32_t c = 0;
      if (!p.w && !__any_sync(0xffffffffu, look)) {
        c = (uint32_t)sv.y;
      } else {
        // 32 entries at a time: lane j loads entry j, the warp broadcasts them
        // and each lane tests its own tree, in row order; the preorder numbers
        // of eight neighbours are loaded before any is tested, so eight loads
        // are in flight (a neighbour past the row's end reads as inside)
        for (int32_t eb = 0; eb < sv.y; eb += 32) {
          const int32_t m = min(32, sv.y - eb);
          if (eb > 0) {
            uj = lane < m ? __ldg(p.colidx + e0 + eb + lane) : 0;
            wj = (p.w && lane < m) ? __ldg(p.w + e0 + eb + lane) : 0.f;
          }
          for (int k0 = 0; k0 < m; k0 += 8) {
            int32_t tu[8];
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
              const int32_t u = __shfl_sync(0xffffffffu, uj, (k0 + kk) & 31);
              tu[kk] = k0 + kk < m ? lo - 1 : lo;
              if (look && k0 + kk < m) tu[kk] = p.tin[VT(lane, u)];
            }
            if (p.w) {
#pragma unroll
              for (int kk = 0; kk < 8; ++kk) {
                const float wk = __shfl_sync(0xffffffffu, wj, (k0 + kk) & 31);
                if (tu[kk] < lo || tu[kk] >= hi) s = __dadd_rn(s, (double)wk);
              }
            } else {
#pragma unroll
              for (int kk = 0; kk < 8; ++kk) c += (uint32_t)(tu[kk] - lo) >= (uint32_t)(hi - lo) ? 1u : 0u;
            }
          }
        }
      }
      if (p.w || p.rowptr[v + 1] - p.rowptr[v] <= RB_SEG) finish(v, s, c);
      else if (on && c) atomicAdd(&p.outc[VT(lane, v)], c);
    }
  }
  grid.sync();

  // ---- rows of several segments, and empty rows ----
  for (int64_t v0 = gwarp * 32; v0 < n; v0 += nwarps * 32) {
    const int64_t d = v0 + lane < n ? p.rowptr[v0 + lane + 1] - p.rowptr[v0 + lane] : 1;
    for (unsigned left = __ballot_sync(0xffffffffu, d == 0 || (!p.w && d > RB_SEG)); left != 0u; left &= left - 1u) {
      const int k = __ffs(left) - 1;
      const int32_t v = (int32_t)v0 + k;
      const bool counted = __shfl_sync(0xffffffffu, d, k) > 0;
      finish(v, 0.0, on && counted ? p.outc[VT(lane, v)] : 0u);
    }
  }
#undef VT
}

// Fixed-point value of 1 / (1 + alpha c) for every count c = 0..cmax of
// outside neighbours (unweighted graphs, one alpha), with the FP64 steps of
// the per-tree formula, so a table lookup gives the same bits.
__global__ void k_rb_table(double alpha, int32_t cmax, uint64_t* __restrict__ qtab) {
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c <= cmax; c += (int64_t)gridDim.x * blockDim.x) {
    const double val = __ddiv_rn(1.0, __dadd_rn(1.0, __dmul_rn(alpha, (double)c)));
    qtab[c] = (uint64_t)__dadd_rn(__dmul_rn(val, (double)(1ull << RB_FRAC)), 0.5);
  }
}

__global__ void k_rb_diag(int32_t n, const uint64_t* __restrict__ acc, double denom, double* __restrict__ diag) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    diag[v] = __ddiv_rn((double)acc[v], denom);
}

// Segments per row: unweighted rows split every RB_SEG entries (their
// integer counts add up exactly); weighted rows stay whole so that each
// tree's sum keeps the row order.  cnt has n + 1 entries, the last 0.
__global__ void k_seg_count(int32_t n, const int64_t* __restrict__ rowptr, bool weighted, uint32_t* __restrict__ cnt) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v <= n; v += (int64_t)gridDim.x * blockDim.x) {
    uint32_t c = 0;
    if (v < n) {
      const int64_t d = rowptr[v + 1] - rowptr[v];
      c = weighted ? (d > 0 ? 1u : 0u) : (uint32_t)((d + RB_SEG - 1) / RB_SEG);
    }
    cnt[v] = c;
  }
}

__global__ void k_seg_fill(int32_t n, const uint32_t* __restrict__ cnt, const uint32_t* __restrict__ off,
                           const int64_t* __restrict__ rowptr, bool weighted, int4* __restrict__ segs) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t o = off[v];
    const int64_t r0 = rowptr[v], r1 = rowptr[v + 1];
    for (uint32_t k = 0; k < cnt[v]; ++k) {
      const int64_t e0 = r0 + (int64_t)k * RB_SEG;
      const int32_t m = (int32_t)(weighted ? r1 - r0 : std::min<int64_t>(RB_SEG, r1 - e0));
      segs[o + k] = make_int4((int32_t)v, m, (int32_t)(uint32_t)e0, (int32_t)(uint32_t)((uint64_t)e0 >> 32));
    }
  }
}

}  // namespace

}  // namespace fcx

using namespace fcx;

// Chunks of up to 32 trees through k_rb<mode>: mode 0 adds the
// Rao-Blackwellised values to acc (uint64), mode 1 the path sums S_T(v) to
// acc (int64).
static fc_status tree_chunks(fc_graph* g, int mode, int32_t alpha_idx, const int32_t* parents, int64_t T, void* acc,
                             cudaStream_t st, const char* who) {
  const int32_t n = g->n;
  int dev = g->device, nsm = 0, coop = 0, per_sm = 0;
  FC_CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  FC_CK(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
  if (!coop) {
    set_error(std::string(who) + ": the device does not support cooperative launches");
    return FC_ECUDA;
  }
  const void* kern = mode == 0 ? (const void*)k_rb<0> : (const void*)k_rb<1>;
  FC_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, RB_T, 0));
  const int grid = std::max(1, per_sm) * nsm;  // every CTA resident: required by the grid barriers
  // trees per chunk: one per lane, 28 bytes of scratch per (tree, vertex)
  // within a sixteenth of the device (1 to 16 GB), flat ids below 2^31
  const int64_t budget = std::max<int64_t>(1ll << 30, std::min<int64_t>(16ll << 30, (int64_t)(g->device_bytes / 16)));
  const int64_t cap = std::max<int64_t>(1, std::min<int64_t>(budget / (28ll * (n + 1)),
                                                             ((int64_t)1 << 31) / ((int64_t)n + 1) - 1));
  const int64_t Tc_max = std::min<int64_t>(std::min<int64_t>(T, RB_TMAX), cap);
  const size_t N = (size_t)Tc_max * n;
  const int64_t seg_max = (int64_t)n + g->nnz / RB_SEG + 1;  // bound on the number of segments
  char* ws = nullptr;
  const size_t bytes = N * 8 * 2 + N * 4 * 3 + 32 + RB_TMAX * 4 + ((size_t)n + 1) * 8 + (size_t)seg_max * 16 +
                       ((size_t)g->max_deg + 1) * 8 + 256 * 16;
  FC_CK(cudaMallocAsync((void**)&ws, bytes, st));
  auto carve = [&](size_t b) {
    char* r = ws;
    ws += (b + 255) & ~(size_t)255;
    return r;
  };
  char* base = ws;
  RBParams p;
  p.n = n;
  p.rowptr = g->rowptr;
  p.colidx = g->colidx;
  p.w = g->w;
  p.alpha = g->alphas[alpha_idx];
  p.alpha_v = g->num_graphs > 0 ? g->alpha_v : nullptr;
  p.acc = mode == 0 ? (uint64_t*)acc : nullptr;
  p.racc = mode == 1 ? (int64_t*)acc : nullptr;
  p.root = mode == 1 ? g->root : -1;
  p.bpar = g->bpar;
  p.binv = g->binv;
  p.word = (unsigned long long*)carve(N * 8);
  p.jw = (unsigned long long*)carve(N * 8);
  p.size = (int32_t*)carve(N * 4);
  p.tin = (int32_t*)carve(N * 4);
  p.outc = (uint32_t*)carve(N * 4);
  p.pvm = (int32_t*)p.outc;  // resistance mode: the tree parents, vertex-major
  p.ctr = (uint32_t*)carve(32 + RB_TMAX * 4);
  p.tsum = p.ctr + 8;
  const bool table = mode == 0 && g->w == nullptr && g->num_graphs == 0;
  uint64_t* qtab = table ? (uint64_t*)carve(((size_t)g->max_deg + 1) * 8) : nullptr;
  p.qtab = qtab;
  uint32_t* scnt = (uint32_t*)carve(((size_t)n + 1) * 4);
  uint32_t* soff = (uint32_t*)carve(((size_t)n + 1) * 4);
  int4* segs = (int4*)carve((size_t)seg_max * 16);
  ws = base;
  p.segs = segs;
  p.nseg = soff + n;
  if (mode == 0) {  // row segments (the resistance mode reads no rows)
    const unsigned b = (unsigned)std::min<int64_t>(((int64_t)n + 256) / 256, (int64_t)nsm * 16);
    k_seg_count<<<b, 256, 0, st>>>(n, g->rowptr, g->w != nullptr, scnt);
    FC_LAUNCHED();
    const fc_status r = exclusive_scan(scnt, soff, (int64_t)n + 1, st);
    if (r != FC_OK) {
      FC_CK(cudaFreeAsync(base, st));
      return r;
    }
    k_seg_fill<<<b, 256, 0, st>>>(n, scnt, soff, g->rowptr, g->w != nullptr, segs);
    FC_LAUNCHED();
    if (table) {
      const unsigned bt = (unsigned)std::min<int64_t>(((int64_t)g->max_deg + 256) / 256, (int64_t)nsm * 4);
      k_rb_table<<<bt, 256, 0, st>>>(p.alpha, g->max_deg, qtab);
      FC_LAUNCHED();
    }
  }
  fc_status status = FC_OK;
  for (int64_t t0 = 0; t0 < T && status == FC_OK; t0 += Tc_max) {
    const int32_t Tc = (int32_t)std::min<int64_t>(Tc_max, T - t0);
    p.Tc = Tc;
    p.parents = parents + (size_t)t0 * n;
    FC_CK(cudaMemsetAsync(p.word, 0, (size_t)Tc * n * 8, st));
    FC_CK(cudaMemsetAsync(p.ctr, 0, 32 + RB_TMAX * 4, st));
    void* args[] = {&p};
    FC_CK(cudaLaunchCooperativeKernel(kern, dim3(grid), dim3(RB_T), args, 0, st));
    FC_LAUNCHED();
    uint32_t herr = 0;
    FC_CK(cudaMemcpyAsync(&herr, p.ctr + 2, 4, cudaMemcpyDeviceToHost, st));
    FC_CK(cudaStreamSynchronize(st));
    if (herr != 0) {
      set_error(std::string(who) + (mode == 0 ? ": parents do not form spanning trees of G* rooted at u* = n"
                                              : ": parents do not form spanning trees of G rooted at the pivot"));
      status = FC_EINVAL;
    }
  }
  FC_CK(cudaFreeAsync(base, st));
  return status;
}

extern "C" fc_status fc_rb_accumulate(fc_graph* g, int32_t alpha_idx, const int32_t* parents, int64_t T,
                                      uint64_t* acc, void* stream) {
  if (g == nullptr || parents == nullptr || acc == nullptr || T < 0 || alpha_idx < 0 ||
      alpha_idx >= g->n_alpha) {
    set_error("fc_rb_accumulate: bad argument");
    return FC_EINVAL;
  }
  if (T == 0) return FC_OK;
  return tree_chunks(g, 0, alpha_idx, parents, T, acc, (cudaStream_t)stream, "fc_rb_accumulate");
}

extern "C" fc_status fc_resistance_accumulate(fc_graph* g, const int32_t* parents, int64_t T, int64_t* acc,
                                              void* stream) {
  if (g == nullptr || parents == nullptr || acc == nullptr || T < 0) {
    set_error("fc_resistance_accumulate: bad argument");
    return FC_EINVAL;
  }
  if (g->root < 0 || g->bpar == nullptr) {
    set_error("fc_resistance_accumulate: needs a graph from fc_build_rooted");
    return FC_EINVAL;
  }
  if (T == 0) return FC_OK;
  return tree_chunks(g, 1, 0, parents, T, acc, (cudaStream_t)stream, "fc_resistance_accumulate");
}

extern "C" fc_status fc_rb_diag(const uint64_t* acc, int32_t n, int64_t T, double* diag_out, void* stream) {
  if (acc == nullptr || diag_out == nullptr || n < 1 || T < 1) {
    set_error("fc_rb_diag: bad argument");
    return FC_EINVAL;
  }
  cudaStream_t st = (cudaStream_t)stream;
  const double denom = (double)(1ull << RB_FRAC) * (double)T;  // exact: a power of two times T
  k_rb_diag<<<(unsigned)std::min<int64_t>((n + 255) / 256, 152 * 16), 256, 0, st>>>(n, acc, denom, diag_out);
  FC_LAUNCHED();
  return FC_OK;
}
