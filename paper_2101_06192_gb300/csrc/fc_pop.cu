// Wilson sampler by parallel cycle popping (Propp-Wilson): the trees of
// Algorithm 2 without walkers that claim vertices.
//
// The random stacks fix the tree: whatever the order in which cycles of the
// current tops are popped, the same cycles are popped and the same tops remain
// (the abelian property that also lets the walker kernels interleave).  So
// instead of walking from start vertices and claiming every vertex of a path,
// this sampler draws the top of EVERY vertex first (one coalesced pass) and
// then looks for the cycles of that functional graph, which are few: on a
// heavy-tailed graph of mean degree 16 about 5% of the vertices lie on one.
//
// A window is a set of trees ("rows": (alpha index, tree) pairs).  One 32-bit
// word per vertex and row: the vertex selected by the current top (n = u*) in
// 29 bits, RED (redrawn at least once: its entry count K is valid) and two
// ACT flags (redrawn in the last round, by the round's parity).  A window runs
// through phases separated by barriers:
//
//   draw    entry 0 of every vertex
//   walk    the cycles of the current tops; tops do not change.  A walk from v
//           follows the words until it reaches u*, goes round a cycle without
//           v (Brent's cycle detection) or returns to v.  In the first round
//           every vertex walks and stops at any vertex below v, so a cycle is
//           found by its smallest vertex alone, and most walks end at once; in
//           later rounds only the vertices redrawn in the last one walk (a new
//           cycle has to hold one of them) and stop at redrawn vertices below
//           v, so a cycle is found by its smallest redrawn vertex alone.  The
//           finder goes round again and appends the cycle's vertices to the
//           next round's list.
//   redraw  every listed vertex takes its next stack entry
//
// until a walk phase finds no cycle.  No locks and no state to clear; a top
// that selects u* is final (it is never on a cycle), so R, C and the
// departures are counted where entries are drawn.  A tree of a batch's graph is
// complete when its last cycle is listed for its redraw: every listing stamps it.
//
// The CTAs of one cooperative launch form teams with their own barriers; each
// team takes its own windows, so while one team waits for its longest walk (a
// chain of dependent loads) the others fill the SMs.
//
// What bounds it (GB300, BA n = 2^20, mean degree 16; 160 trees, phases timed as
// launches of their own): drawing 3.7 us per tree, issue (131 warp instructions
// per 32 vertices, most of them Philox); first walks 6.0 us, latency of 0.7 n
// dependent 4-byte gathers (110 G/s of the 290 G/s that independent gathers
// reach); redraws 3.9 us, DRAM (290 bytes per listed vertex at 4.8 TB/s: word,
// row info and target lie in different sectors); later rounds 5 us.  The walker
// kernels took 41 us per tree, 570 warp instructions per iteration.
#include <cooperative_groups.h>

#include <algorithm>

#include "fc_wilson_common.cuh"

namespace fcx {

namespace {

constexpr uint32_t PW_RED = 1u << 29;
constexpr uint32_t PW_ACT = 1u << 30;  // shifted by the round's parity
constexpr uint32_t PW_ID = PW_RED - 1u;
constexpr uint32_t PW_NONE = 0xffffffffu;
constexpr int PK_T = 256;      // threads per CTA
constexpr int PK_W = PK_T / 32;
constexpr int PK_CHUNK = 256;  // vertices of one row looked at by a warp at a time
constexpr int PK_RING = 512;   // candidates waiting per warp (a power of two, over PK_CHUNK + 32)
constexpr int PK_OWN = 64;     // finders noted by a warp
constexpr int PK_STEPS = 4;    // walk steps between two looks for idle lanes

struct PopParams {
  int32_t n;
  int64_t nnz;
  const uint4* rowinfo;   // [n_alpha][n] {row offset, degree, T lo, T hi}
  const int32_t* colidx;  // [nnz]
  const uint64_t* B;      // [n_alpha][nnz] slot thresholds, or null (unweighted)
  int64_t tau, tree_offset;
  uint32_t key0, key1;
  int64_t total;          // rows of the call
  int32_t wrows;          // rows per window
  int32_t teams, ctas;    // teams, CTAs per team
  uint32_t ld;            // words per row (a multiple of 4)
  uint32_t ld_mul, ld_shift;  // division by ld (row_of_item)
  uint32_t* F;            // [teams][wrows][ld] tops
  uint32_t* K;            // [teams][wrows][ld] entries popped (RED vertices)
  uint32_t* L;            // [teams][2][wrows * ld] listed vertices (row * ld + v)
  uint32_t* ctl;          // [teams][32] barrier and list counts (zeroed)
  uint32_t* R;
  uint32_t* C;
  unsigned long long* visits;
  unsigned long long* steps;  // single graphs: [row]; batches: [graph][tree]
  int32_t* parents;           // [row][n] or null
  int32_t num_graphs;         // 0 = single graph
  const int64_t* voff;
  const int32_t* gid;
  unsigned long long* item_ns;
  uint32_t* err;
  unsigned long long* stats;  // [0] pops, [1] departures
  uint32_t max_iters;
};

enum { CTL_ARRIVE = 0, CTL_GEN = 8, CTL_COUNT = 16 };  // words of a team's control block
constexpr uint32_t GEN_ABORT = 0x80000000u;
constexpr uint32_t POP_SPIN = 1u << 23;  // polls of a barrier before it gives up

// Tops within a walk phase, where nothing writes them: cached in L1 (the
// barrier's acquire drops lines of the phases before; a team of one CTA writes
// its tops from the same SM, and the block's barrier orders its threads).
__device__ __forceinline__ uint32_t ld_top(const uint32_t* a) {
  uint32_t v;
  asm volatile("ld.global.ca.u32 %0, [%1];" : "=r"(v) : "l"(a) : "memory");
  return v;
}

// Barrier of a team (all CTAs of the launch are resident).  Returns true when
// the launch is to be left: the last CTA to arrive reads the error word for
// all of them, so they leave together.  A team of one CTA looks at it every 16th
// time only (n = 2, three alphas x 50 trees, some 200 rounds each: 451
// -> 279 us a call, the walker kernels 342).
template <bool ONE>
__device__ __forceinline__ bool team_sync(uint32_t* ctl, int ctas, uint32_t& gen, const uint32_t* err) {
  __shared__ uint32_t sh_abort;
  if (ONE && (++gen & 15u) != 0u) {
    __syncthreads();
    return false;
  }
  __syncthreads();
  if (ONE) {
    if (threadIdx.x == 0) sh_abort = *(volatile const uint32_t*)err;
    __syncthreads();
    return sh_abort != 0u;
  }
  if (threadIdx.x == 0) {
    ++gen;
    uint32_t old, g = 0;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(old) : "l"(ctl + CTL_ARRIVE) : "memory");
    if (old + 1u == gen * (uint32_t)ctas) {
      g = gen | (*(volatile const uint32_t*)err != 0u ? GEN_ABORT : 0u);
      asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(ctl + CTL_GEN), "r"(g) : "memory");
    } else {
      uint32_t i = 0;
      for (; i < POP_SPIN; ++i) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(g) : "l"(ctl + CTL_GEN) : "memory");
        if ((g & ~GEN_ABORT) >= gen) break;
        __nanosleep(32);
      }
      if (i == POP_SPIN) {  // a CTA of the team never came: leave with an error
        atomicOr((uint32_t*)err, ERR_TIMEOUT);
        g = GEN_ABORT;
      }
    }
    sh_abort = g & GEN_ABORT;
  }
  __syncthreads();
  return sh_abort != 0u;
}

// alpha index and tree of row r of the call
__device__ __forceinline__ void row_of(const PopParams& p, int64_t g, int32_t* a, int64_t* t) {
  if (g < p.tau) {  // one alpha, or the first of several
    *a = 0;
    *t = g;
  } else {
    const int64_t q = g / p.tau;
    *a = (int32_t)q;
    *t = g - q * p.tau;
  }
}

// row of a listed vertex (item row * ld + v): a multiply and a shift instead
// of a division (exact for items below 2^32: floor(i / d) by the round-up
// method with a 33-bit multiplier folded into an add)
__device__ __forceinline__ uint32_t row_of_item(const PopParams& p, uint32_t it) {
  const uint32_t h = __umulhi(it, p.ld_mul);
  return (((it - h) >> 1) + h) >> p.ld_shift;
}

// first slot j of a row of d entries with u < b[j] (b[d - 1] = 2^53)
__device__ __forceinline__ uint32_t slot_search(const uint64_t* b, uint32_t d, uint64_t u) {
  uint32_t lo = 0, hi = d - 1u;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (u < __ldg(b + mid)) hi = mid;
    else lo = mid + 1u;
  }
  return lo;
}

// draw: entry 0 of every vertex in rows [g0, g0 + rows); a thread per vertex,
// the rows in a loop (row info, and a short row's thresholds, in registers;
// the targets of the row stay in L1).
template <bool WGT, bool BAT>
__device__ void pop_draw(const PopParams& p, uint32_t* F, int64_t g0, int32_t rows, int cta) {
  const int32_t nv = (p.n + PK_T - 1) / PK_T;
  // rows per task: as many as leave two tasks per CTA
  int32_t rg = rows;
  while (rg > 1 && (int64_t)nv * ((rows + rg - 1) / rg) < 2 * (int64_t)p.ctas) rg = (rg + 1) >> 1;
  const int32_t ng = (rows + rg - 1) / rg;
  for (int64_t task = cta; task < (int64_t)nv * ng; task += p.ctas) {
    const int32_t grp = (int32_t)(task / nv);
    const int32_t v = (int32_t)(task - (int64_t)grp * nv) * PK_T + (int32_t)threadIdx.x;
    if (v >= p.n) continue;
    int32_t r = grp * rg;
    const int32_t r1 = min(r + rg, rows);
    int32_t a;
    int64_t t;
    row_of(p, g0 + r, &a, &t);
    int32_t gi = 0, nl = p.n;
    bool lead = v == 0 && p.steps != nullptr;
    if (BAT && p.steps != nullptr) {
      gi = p.gid[v];
      lead = p.voff[gi] == v;
      nl = (int32_t)(p.voff[gi + 1] - v);
    }
    while (r < r1) {
      // the rows of one alpha
      const int32_t re = (int32_t)min((int64_t)r1, (int64_t)r + (p.tau - t));
      const uint4 ri = __ldg(p.rowinfo + (size_t)a * p.n + v);
      const uint64_t T = (uint64_t)ri.z | ((uint64_t)ri.w << 32);
      const uint64_t* b = WGT ? p.B + (size_t)a * p.nnz + ri.x : nullptr;
      const int32_t* col = p.colidx + ri.x;
      uint64_t bv[7];
      if (WGT) {
#pragma unroll
        for (int j = 0; j < 7; ++j) bv[j] = (ri.y <= 8u && j + 1 < (int)ri.y) ? __ldg(b + j) : ~0ull;
      }
      uint32_t cnt = 0;
      const int32_t rb = r;
      const uint32_t tb = (uint32_t)(p.tree_offset + t) - (uint32_t)rb;
#pragma unroll 4
      for (; r < re; ++r) {
        const uint4 o = philox4x32_10(0u, (uint32_t)v, tb + (uint32_t)r, (uint32_t)a, p.key0, p.key1);
        const uint64_t u = stack_u53(o);
        uint32_t w = (uint32_t)p.n;
        if (u < T) {
          ++cnt;
        } else {
          uint32_t slot;
          if (!WGT) {
            slot = __umulhi(o.z, ri.y);
          } else if (ri.y <= 8u) {
            slot = 0;
#pragma unroll
            for (int j = 0; j < 7; ++j) slot += u >= bv[j] ? 1u : 0u;
          } else {
            slot = slot_search(b, ri.y, u);
          }
          w = (uint32_t)__ldg(col + slot);
        }
        F[(size_t)r * p.ld + v] = w;
      }
      if (cnt) {
        atomicAdd(p.R + (size_t)a * p.n + v, cnt);
        if (p.C != nullptr) atomicAdd(p.C + (size_t)a * p.n + v, cnt);
      }
      if (p.visits != nullptr) atomicAdd(p.visits + (size_t)a * p.n + v, (unsigned long long)(r - rb));
      if (lead) {
        unsigned long long* s = p.steps + (BAT ? (size_t)gi : (size_t)a) * p.tau + (size_t)t;
        for (int32_t q = rb; q < r; ++q) s[q - rb] = (unsigned long long)nl;
      }
      ++a;
      t = 0;
    }
  }
}

// redraw: the next stack entry of every listed vertex; the last round's ACT
// flags are cleared (a vertex in both lists ends with the new word either way)
template <bool WGT, bool BAT>
__device__ void pop_redraw(const PopParams& p, uint32_t* F, uint32_t* K, const uint32_t* list, uint32_t cnt,
                           const uint32_t* old, uint32_t oldcnt, int par, int64_t g0, int cta) {
  const uint32_t stride = (uint32_t)p.ctas * PK_T;
  WParams sp;
  sp.B = WGT ? p.B : nullptr;
  sp.nnz = p.nnz;
  for (uint32_t i = (uint32_t)cta * PK_T + threadIdx.x; i < oldcnt; i += stride)
    atomicAnd(F + __ldcg(old + i), ~(PW_ACT << (par ^ 1)));
  for (uint32_t i = (uint32_t)cta * PK_T + threadIdx.x; i < cnt; i += stride) {
    const uint32_t it = __ldcg(list + i);
    const uint32_t r = row_of_item(p, it), v = it - r * p.ld;
    int32_t a;
    int64_t t;
    row_of(p, g0 + r, &a, &t);
    const uint4 ri = __ldg(p.rowinfo + (size_t)a * p.n + v);
    uint32_t k = 1;
    if (__ldcg(F + it) & PW_RED) k = __ldcg(K + it) + 1u;
    if (k >= (uint32_t)K_MASK) atomicOr(p.err, ERR_OVERFLOW);
    const uint4 o = philox4x32_10(k, v, (uint32_t)(p.tree_offset + t), (uint32_t)a, p.key0, p.key1);
    uint32_t e = 0, w = (uint32_t)p.n;
    if (select_edge(sp, a, ri, o, &e)) {
      w = (uint32_t)__ldg(p.colidx + e);
      K[it] = k;
    } else {
      atomicAdd(p.R + (size_t)a * p.n + v, 1u);
    }
    F[it] = w | PW_RED | (PW_ACT << par);
    if (p.visits != nullptr) atomicAdd(p.visits + (size_t)a * p.n + v, 1ull);
  }
}

// The vertices of the cycles whose finders are listed in own[0, cnt), a lane
// per cycle: round once for the lengths, once more to append the vertices (the
// walk that found the cycle left its tops in L1).
template <bool BAT>
__device__ uint32_t pop_list_cycles(const PopParams& p, const uint32_t* F, const uint32_t* own, int cnt, uint32_t* out,
                                    uint32_t* outcnt, int64_t g0) {
  const int lane = threadIdx.x & 31;
  uint32_t rb = 0, v = 0, len = 0, row = 0;
  int32_t gi = 0;
  const unsigned long long ns = BAT ? global_ns() : 0ull;
  if (lane < cnt) {
    const uint32_t it = own[lane];
    row = row_of_item(p, it);
    rb = row * p.ld;
    v = it - rb;
    if (BAT) gi = __ldg(p.gid + v);  // needed at the end
    uint32_t x = v;
    do {
      x = ld_top(F + (rb + x)) & PW_ID;
      ++len;
    } while (x != v);
  }
  __syncwarp();
  uint32_t s = len;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(FULL, s, o);
    if (lane >= o) s += y;
  }
  uint32_t b = 0;
  if (lane == 31) b = atomicAdd(outcnt, s);
  b = __shfl_sync(FULL, b, 31);
  if (len) {
    uint32_t* o = out + (b + s - len);
    uint32_t x = v;
    do {
      *o++ = rb + x;
      x = ld_top(F + (rb + x)) & PW_ID;
    } while (x != v);
    if (p.steps != nullptr) {
      int32_t a;
      int64_t t;
      row_of(p, g0 + row, &a, &t);
      atomicAdd(p.steps + (BAT ? (size_t)gi : (size_t)a) * p.tau + (size_t)t,
                (unsigned long long)len);
    }
    // the tree's completion time, unless it has a cycle in a later round too (any
    // of the stamps that it gets in this phase will do: they are moments apart).
    // 256 uneven graphs, 64 trees on GB300: a stamp per cycle with the graph's
    // number loaded ahead costs 1.3% of a call, one per redrawn vertex 3 to 5%
    if (BAT) p.item_ns[(size_t)gi * p.tau + (size_t)(g0 + row)] = ns;
  }
  __syncwarp();
  return len;
}

// walk: FIRST: every vertex of the window, else the listed ones (cnt of them,
// ACT flag of parity par).  Vertices of the cycles found are appended to out.
// Returns this thread's count of them.
//
// A warp's lanes walk independently and are bound by the latency of the
// dependent loads, so every lane is kept on a walk: candidates wait in a ring
// in shared memory, and the words of the next unit (PK_CHUNK vertices of a
// row, or 32 listed vertices) are loaded while the lanes walk.
template <bool FIRST, bool BAT>
__device__ uint32_t pop_walk(const PopParams& p, const uint32_t* F, const uint32_t* list, uint32_t cnt, int par,
                             uint32_t* out, uint32_t* outcnt, int64_t g0, int32_t rows, int cta, uint2* q,
                             uint32_t* own) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const uint32_t n = (uint32_t)p.n, ld = p.ld;
  const uint32_t act = PW_ACT << par;
  const uint32_t cpr = (n + PK_CHUNK - 1) / PK_CHUNK;  // chunks per row
  const uint32_t units = FIRST ? cpr * (uint32_t)rows : (cnt + 31u) / 32u;
  const uint32_t nw = (uint32_t)p.ctas * PK_W;
  uint32_t unit = (threadIdx.x >> 5) * (uint32_t)p.ctas + (uint32_t)cta;  // the unit whose words are in flight
  uint32_t qh = 0, qn = 0;  // warp-uniform: ring [qh, qn) of candidates {item, selected vertex}
  int no = 0;               // finders noted
  bool walk = false;
  uint32_t rb = 0, v = 0, x = 0, tort = 0, iters = 0, pops = 0;

  // FIRST: words of the unit in flight and its place; else its items and
  // words, and the items of the unit after it
  uint4 w4[2];
  uint32_t ub = 0, v0 = 0, it1 = PW_NONE, w1 = 0, it2 = PW_NONE;
  auto load_chunk = [&]() {
    if (unit < units) {
      const uint32_t row = unit / cpr;
      ub = row * ld;
      v0 = (unit - row * cpr) * PK_CHUNK + lane * 4;
#pragma unroll
      for (int i = 0; i < 2; ++i)
        w4[i] = v0 + i * 128 < n ? __ldcg(reinterpret_cast<const uint4*>(F + ub + v0 + i * 128)) : make_uint4(n, n, n, n);
    }
  };
  auto load_item = [&](uint32_t u) {
    const uint32_t i = u * 32u + lane;
    return u < units && i < cnt ? __ldcg(list + i) : PW_NONE;
  };
  if (FIRST) {
    load_chunk();
  } else {
    it1 = load_item(unit);
    it2 = unit + nw < units ? load_item(unit + nw) : PW_NONE;
    if (it1 != PW_NONE) w1 = ld_top(F + it1);
  }
  for (;;) {
    // ---- the arrived unit's candidates, while the ring runs low ----
    while (qn - qh < 32u && unit < units) {
      if (FIRST) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const uint32_t vv = v0 + (i >> 2) * 128 + (i & 3);
          const uint4 ww = w4[i >> 2];
          const uint32_t w = (i & 3) == 0 ? ww.x : (i & 3) == 1 ? ww.y : (i & 3) == 2 ? ww.z : ww.w;
          const bool cand = vv < n && w != n && w > vv;  // a walk that does not stop at once
          const unsigned m = __ballot_sync(FULL, cand);
          if (cand) q[(qn + __popc(m & lt)) & (PK_RING - 1)] = make_uint2(ub + vv, w);
          qn += __popc(m);
        }
        unit += nw;
        load_chunk();
      } else {
        const uint32_t w = w1 & PW_ID;
        const bool cand = it1 != PW_NONE && w != n;
        const unsigned m = __ballot_sync(FULL, cand);
        if (cand) q[(qn + __popc(m & lt)) & (PK_RING - 1)] = make_uint2(it1, w);
        qn += __popc(m);
        unit += nw;
        it1 = it2;
        if (it1 != PW_NONE) w1 = ld_top(F + it1);
        it2 = unit + nw < units ? load_item(unit + nw) : PW_NONE;
      }
      __syncwarp();
    }
    // ---- idle lanes take candidates ----
    const unsigned idle = __ballot_sync(FULL, !walk);
    if (idle) {
      const uint32_t r = (uint32_t)__popc(idle & lt);
      if (!walk && r < qn - qh) {
        const uint2 cw = q[(qh + r) & (PK_RING - 1)];
        rb = row_of_item(p, cw.x) * ld;
        v = cw.x - rb;
        x = tort = cw.y;
        iters = 0;
        walk = true;
      }
      __syncwarp();
      qh += min(qn - qh, (uint32_t)__popc(idle));
      if (!__any_sync(FULL, walk)) {
        if (unit < units) continue;
        break;
      }
    }
    // ---- a few steps ----
    bool found = false;
#pragma unroll
    for (int s = 0; s < PK_STEPS; ++s) {
      if (walk) {
        const uint32_t w = ld_top(F + (rb + x));
        const uint32_t y = w & PW_ID;
        bool stop = y == n || y == tort;
        if (FIRST) stop |= y < v;
        else stop |= (w & act) != 0u && x < v;
        found = !stop && y == v;
        walk = !stop && y != v;
        x = y;
        ++iters;
        if ((iters & (iters - 1u)) == 0u) tort = y;  // Brent: a new reference at every power of two
      }
    }
    if (iters > p.max_iters) {
      atomicOr(p.err, ERR_TIMEOUT);
      walk = false;
    }
    const unsigned m = __ballot_sync(FULL, found);
    if (m) {
      if (found) own[no + __popc(m & lt)] = rb + v;
      no += __popc(m);
      __syncwarp();
      if (no >= 32) {
        pops += pop_list_cycles<BAT>(p, F, own + (no - 32), 32, out, outcnt, g0);
        no -= 32;
        __syncwarp();
      }
    }
  }
  if (no) pops += pop_list_cycles<BAT>(p, F, own, no, out, outcnt, g0);
  __syncwarp();
  return pops;
}

// completion times of a batch's trees in rows [g0, g0 + rows): now
__device__ void pop_stamp(const PopParams& p, int64_t g0, int32_t rows, int cta) {
  const unsigned long long ns = global_ns();
  const int64_t len = (int64_t)rows * p.num_graphs;
  for (int64_t i = (int64_t)cta * PK_T + threadIdx.x; i < len; i += (int64_t)p.ctas * PK_T)
    p.item_ns[(i / rows) * p.tau + g0 + i % rows] = ns;
}

__device__ __forceinline__ void pop_stats(const PopParams& p, uint32_t pops) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) pops += __shfl_xor_sync(FULL, pops, o);
  if ((threadIdx.x & 31) == 0 && pops) {
    atomicAdd(&p.stats[0], (unsigned long long)pops);
    atomicAdd(&p.stats[1], (unsigned long long)pops);
  }
}

// BAT: a batch (steps and completion times per graph); ONE: teams of one CTA.
// Templates, because the kernel is at its 64 registers (BA n = 2^20 from CSR, 1024
// trees, whole calls: 24.87 ms with both decided at run time, 24.27 so).
template <bool WGT, bool BAT, bool ONE>
__global__ void __launch_bounds__(PK_T, 4) k_pop(PopParams p) {
  __shared__ uint2 sh_q[PK_W][PK_RING];
  __shared__ uint32_t sh_e[PK_W][PK_OWN];
  const int team = (int)(blockIdx.x / (unsigned)p.ctas), cta = (int)(blockIdx.x % (unsigned)p.ctas);
  const int wid = threadIdx.x >> 5;
  const size_t cap = (size_t)p.wrows * p.ld;
  uint32_t* F = p.F + (size_t)team * cap;
  uint32_t* K = p.K + (size_t)team * cap;
  uint32_t* L = p.L + (size_t)team * 2 * cap;
  uint32_t* ctl = p.ctl + team * 32;
  uint32_t* lc = ctl + CTL_COUNT;  // list counts, by round mod 3
  uint32_t gen = 0, pops = 0;
  const int64_t windows = (p.total + p.wrows - 1) / p.wrows;
  bool quit = false;
  for (int64_t win = team; win < windows; win += p.teams) {
    const int64_t g0 = win * p.wrows;
    const int32_t rows = (int32_t)min((int64_t)p.wrows, p.total - g0);
    pop_draw<WGT, BAT>(p, F, g0, rows, cta);
    if (cta == 0 && threadIdx.x == 0) lc[0] = lc[1] = 0u;
    if ((quit = team_sync<ONE>(ctl, p.ctas, gen, p.err))) break;
    if (BAT) pop_stamp(p, g0, rows, cta);  // complete unless a cycle is found
    uint32_t cnt = 0;
    for (uint32_t rd = 0;; ++rd) {
      // round rd: its list in L[rd & 1] (every vertex for rd = 0)
      uint32_t* nxt = L + (size_t)((rd + 1) & 1u) * cap;
      uint32_t* cur = L + (size_t)(rd & 1u) * cap;
      if (cta == 0 && threadIdx.x == 0) {
        lc[(rd + 2) % 3] = 0u;  // last read two barriers ago
        if (rd > p.max_iters) atomicOr(p.err, ERR_TIMEOUT);
      }
      if (rd == 0) pops += pop_walk<true, BAT>(p, F, cur, 0u, 0, nxt, lc + 1, g0, rows, cta, sh_q[wid], sh_e[wid]);
      else
        pops += pop_walk<false, BAT>(p, F, cur, cnt, (int)(rd & 1u), nxt, lc + (rd + 1) % 3, g0, rows, cta, sh_q[wid],
                                sh_e[wid]);
      if ((quit = team_sync<ONE>(ctl, p.ctas, gen, p.err))) break;
      const uint32_t nc = __ldcg(lc + (rd + 1) % 3);
      if (nc == 0u) break;  // uniform: not written before the next barrier
      pop_redraw<WGT, BAT>(p, F, K, nxt, nc, cur, cnt, (int)((rd + 1) & 1u), g0, cta);
      cnt = nc;
      if ((quit = team_sync<ONE>(ctl, p.ctas, gen, p.err))) break;
    }
    if (quit) break;
    if (p.parents != nullptr) {
      const int64_t len = (int64_t)rows * p.n;
      for (int64_t i = (int64_t)cta * PK_T + threadIdx.x; i < len; i += (int64_t)p.ctas * PK_T) {
        const int64_t r = i / p.n;
        p.parents[g0 * p.n + i] = (int32_t)(F[r * p.ld + (i - r * p.n)] & PW_ID);
      }
      if (BAT) pop_stamp(p, g0, rows, cta);  // the parents are part of the trees
    }
    if ((quit = team_sync<ONE>(ctl, p.ctas, gen, p.err))) break;  // the tops are read before they are drawn again
  }
  pop_stats(p, pops);
}

// What a call starts from, in one launch: a call on a tiny graph is launches.
// n = 3, 1000 trees on GB300, whole calls: 132 us with two clears, a cooperative
// launch and a full barrier per phase, 102 now (the walker kernels: 112).
// (ctl: the barriers of teams of several CTAs)
__global__ void k_pop_begin(unsigned long long* t0_ns, unsigned long long* stats, unsigned long long departures,
                            uint32_t* err, uint32_t* ctl, int words) {
  for (int i = threadIdx.x; i < words; i += blockDim.x) ctl[i] = 0u;
  if (threadIdx.x != 0) return;
  if (err) *err = 0u;
  if (t0_ns) *t0_ns = global_ns();
  stats[0] = 0;
  stats[1] = departures;
  for (int i = 0; i < N_CNT; ++i) stats[2 + i] = 0;  // the walkers' counters
}

}  // namespace

// Tops in flight: larger windows spread the wait for a phase's longest walk
// over more rows, smaller ones stay closer to L2.  Measured on GB300, 4 teams,
// windows of 20 / 40 / 80 / 160 / 400 MB per team: BA n = 2^20, 1024 trees 36.3 /
// 28.3 / 25.0 / 23.7 / 25.8 ms.
constexpr int64_t POP_WINDOW = 640ll << 20;  // bytes of tops, all teams
// Teams: with one CTA per team a barrier costs little and every tree advances
// at its own pace, with one CTA per SM the draws of many trees share a vertex's
// row.  Measured with 4 / 8 / 76 / 608 teams (ms): ER n = 1000, 2000 trees 0.34 /
// 0.32 / 0.29 / 0.24; three alphas x 300 trees of a 128^2 grid 5.6 / 5.0 / 4.1 /
// 3.5; BA 2^18 rooted at its hub (long chains of rounds), 128 trees 8.2 / 7.5 /
// 6.0 / 5.9; R-MAT 2^18, 32 trees 0.43 / 0.42 / 0.43 / 0.43; 256 uneven graphs (2e6
// vertices) x 64 trees 4.95 / 4.78 / 5.13 / 5.11; R-MAT 2^22, 64 trees 5.1 / 5.5 /
// 6.8 / 6.8; BA 2^20, 1024 trees 21.7 / 20.4 / 28.8 / 45.3.
constexpr int32_t POP_MANY_N = 1 << 17;  // every CTA a team up to this size, and for rooted graphs

template <bool ONE>
static const void* pop_fn(const fc_graph* g) {
  if (g->num_graphs > 0)
    return g->weighted ? (const void*)k_pop<true, true, ONE> : (const void*)k_pop<false, true, ONE>;
  return g->weighted ? (const void*)k_pop<true, false, ONE> : (const void*)k_pop<false, false, ONE>;
}

fc_status pop_plan(const fc_graph* g, int64_t total, PopPlan* pl) {
  int nsm = 0, coop = 0, per_sm = g->pop_per_sm.load(std::memory_order_relaxed);
  FC_CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, g->device));
  FC_CK(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, g->device));
  if (per_sm == 0) {  // of the kernel and the device alone
    FC_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, pop_fn<false>(g), PK_T, 0));
    g->pop_per_sm.store(per_sm, std::memory_order_relaxed);
  }
  if (!coop || per_sm < 1) {
    set_error("fc_sample_usts: the device does not support cooperative launches");
    return FC_ECUDA;
  }
  const int64_t ld = ((int64_t)g->n + 3) & ~(int64_t)3;
  const bool many = g->root >= 0 || g->n <= POP_MANY_N;
  pl->teams = (int)std::min<int64_t>(many ? (int64_t)nsm * per_sm : per_sm, total);
  // 16 bytes per vertex and row (top, entry count, two lists) within a quarter of the device
  while (pl->teams > 1 && (size_t)pl->teams * ld * 16 > g->device_bytes / 4) --pl->teams;
  const int64_t cap = std::max<int64_t>(1, POP_WINDOW / pl->teams / (ld * 4));
  pl->wrows = (int32_t)std::max<int64_t>(1, std::min<int64_t>(cap, (total + pl->teams - 1) / pl->teams));
  while (pl->wrows > 1 && (size_t)pl->teams * pl->wrows * ld * 16 > g->device_bytes / 4) pl->wrows = (pl->wrows + 1) / 2;
  // CTAs per team: every SM, fewer when a window is small (a barrier of few CTAs is quicker)
  const int64_t full = (int64_t)nsm * per_sm / pl->teams;
  const int64_t want = ((int64_t)pl->wrows * g->n + 4 * PK_T - 1) / (4 * PK_T);
  pl->ctas = (int)std::max<int64_t>(1, std::min<int64_t>(full, want));
  pl->bytes = (size_t)pl->teams * pl->wrows * ld * 16 + (size_t)pl->teams * 128;
  return FC_OK;
}

fc_status pop_sample(fc_graph* g, const WParams& w, const PopPlan& pl, void* ws, bool reset_err, cudaStream_t st) {
  PopParams p;
  p.n = g->n;
  p.nnz = g->nnz;
  p.rowinfo = g->rowinfo;
  p.colidx = g->colidx;
  p.B = g->weighted ? g->B : nullptr;
  p.tau = w.tau;
  p.tree_offset = w.tree_offset;
  p.key0 = w.key0;
  p.key1 = w.key1;
  p.total = (int64_t)(g->num_graphs > 0 ? 1 : g->n_alpha) * w.tau;
  p.wrows = pl.wrows;
  p.teams = pl.teams;
  p.ctas = pl.ctas;
  p.ld = ((uint32_t)g->n + 3u) & ~3u;
  {
    // floor(i / ld) = ((i - h) / 2 + h) >> (s - 1) with s = ceil(log2 ld) and
    // h = high word of i * (floor(2^32 (2^s - ld) / ld) + 1)
    uint32_t s = 0;
    while ((1ull << s) < p.ld) ++s;
    p.ld_mul = (uint32_t)((((1ull << s) - p.ld) << 32) / p.ld + 1ull);
    p.ld_shift = s - 1u;  // ld >= 4
  }
  const size_t cap = (size_t)pl.teams * pl.wrows * p.ld;
  p.F = (uint32_t*)ws;
  p.K = p.F + cap;
  p.L = p.K + cap;
  p.ctl = p.L + 2 * cap;
  p.R = w.R;
  p.C = w.C;
  p.visits = w.visits;
  p.steps = (unsigned long long*)w.steps;
  p.parents = w.parents;
  p.num_graphs = g->num_graphs;
  p.voff = g->voff;
  p.gid = g->gid;
  p.item_ns = w.item_ns;
  p.err = w.err;
  p.stats = w.stats;
  p.max_iters = w.max_iters;
  k_pop_begin<<<1, 512, 0, st>>>(w.t0_ns, w.stats, (unsigned long long)g->n * (unsigned long long)p.total,
                                 reset_err ? w.err : nullptr, p.ctl, pl.ctas == 1 ? 0 : pl.teams * 32);
  FC_LAUNCHED();
  void* args[] = {&p};
  const dim3 grid((unsigned)(pl.teams * pl.ctas));
  // teams of one CTA wait for no other: no cooperative launch
  FC_CK(pl.ctas == 1 ? cudaLaunchKernel(pop_fn<true>(g), grid, dim3(PK_T), args, 0, st)
                     : cudaLaunchCooperativeKernel(pop_fn<false>(g), grid, dim3(PK_T), args, 0, st));
  FC_LAUNCHED();
  g->last_W = PK_T;
  g->last_regs = 64;
  g->last_grid = pl.teams * pl.ctas;
  g->last_kernel = 5;
  g->last_cluster = 1;
  return FC_OK;
}

}  // namespace fcx
