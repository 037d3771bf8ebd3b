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
// departures are counted where entries are drawn.
//
// The CTAs of one cooperative launch form teams of one CTA per SM with their
// own barriers; each team takes its own windows, so while one team waits for
// its longest walk (a chain of dependent loads) the others fill the SMs.
#include <cooperative_groups.h>

#include <algorithm>

#include "fc_wilson_common.cuh"

namespace fcx {

namespace {

constexpr uint32_t PW_RED = 1u << 29;
constexpr uint32_t PW_ACT = 1u << 30;  // shifted by the round's parity
constexpr uint32_t PW_ID = PW_RED - 1u;
constexpr int PK_T = 256;      // threads per CTA
constexpr int PK_W = PK_T / 32;
constexpr int PK_CHUNK = 256;  // vertices of one row looked at by a warp at a time
constexpr int PK_EMIT = 128;   // listed vertices buffered by a warp

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
// barrier's acquire drops lines of the phases before).
__device__ __forceinline__ uint32_t ld_top(const uint32_t* a) {
  uint32_t v;
  asm volatile("ld.global.ca.u32 %0, [%1];" : "=r"(v) : "l"(a) : "memory");
  return v;
}

// Barrier of a team (all CTAs of the launch are resident).  Returns true when
// the launch is to be left: the last CTA to arrive reads the error word for
// all of them, so they leave together.
__device__ __forceinline__ bool team_sync(uint32_t* ctl, int ctas, uint32_t& gen, const uint32_t* err) {
  __shared__ uint32_t sh_abort;
  __syncthreads();
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

// draw: entry 0 of every vertex in rows [g0, g0 + rows); a thread per vertex,
// the rows in a loop (row info, and a short row's thresholds, in registers;
// the targets of the row stay in L1).
template <bool WGT>
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
    if (p.num_graphs > 0 && p.steps != nullptr) {
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
            uint32_t lo = 0, hi = ri.y - 1u;
            while (lo < hi) {
              const uint32_t mid = (lo + hi) >> 1;
              if (u < __ldg(b + mid)) hi = mid;
              else lo = mid + 1u;
            }
            slot = lo;
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
        unsigned long long* s = p.steps + (p.num_graphs > 0 ? (size_t)gi : (size_t)a) * p.tau + (size_t)t;
        for (int32_t q = rb; q < r; ++q) s[q - rb] = (unsigned long long)nl;
      }
      ++a;
      t = 0;
    }
  }
}

// redraw: the next stack entry of every listed vertex; the last round's ACT
// flags are cleared (a vertex in both lists ends with the new word either way)
__device__ void pop_redraw(const PopParams& p, uint32_t* F, uint32_t* K, const uint32_t* list, uint32_t cnt,
                           const uint32_t* old, uint32_t oldcnt, int par, int64_t g0, int cta) {
  const uint32_t stride = (uint32_t)p.ctas * PK_T;
  WParams sp;
  sp.B = p.B;
  sp.nnz = p.nnz;
  for (uint32_t i = (uint32_t)cta * PK_T + threadIdx.x; i < oldcnt; i += stride)
    atomicAnd(F + __ldcg(old + i), ~(PW_ACT << (par ^ 1)));
  for (uint32_t i = (uint32_t)cta * PK_T + threadIdx.x; i < cnt; i += stride) {
    const uint32_t it = __ldcg(list + i);
    const uint32_t r = it / p.ld, v = it - r * p.ld;
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

// walk: FIRST: every vertex of the window, else the listed ones (cnt of them,
// ACT flag of parity par).  Vertices of the cycles found are appended to out.
// Returns this thread's count of them.
template <bool FIRST>
__device__ uint32_t pop_walk(const PopParams& p, const uint32_t* F, const uint32_t* list, uint32_t cnt,
                             int par, uint32_t* out, uint32_t* outcnt, int64_t g0, int32_t rows, int cta, uint2* q,
                             uint32_t* em) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const uint32_t n = (uint32_t)p.n, ld = p.ld;
  const uint32_t act = PW_ACT << par;
  const uint32_t cpr = (n + PK_CHUNK - 1) / PK_CHUNK;  // chunks per row
  const uint64_t units = FIRST ? (uint64_t)cpr * (uint32_t)rows : ((uint64_t)cnt + 31) / 32;
  const uint64_t nw = (uint64_t)p.ctas * PK_W;
  uint64_t unit = (uint64_t)(threadIdx.x >> 5) * p.ctas + cta;
  int qh = 0, qn = 0, ne = 0;  // warp-uniform: queue [qh, qn), buffered vertices
  uint32_t qb = 0;             // FIRST: row base of the queue
  bool walk = false, emit = false;
  uint32_t rb = 0, v = 0, x = 0, tort = 0, lam = 0, pw = 0, iters = 0, clen = 0, pops = 0;
  for (;;) {
    // ---- idle lanes take the next vertices ----
    unsigned idle = __ballot_sync(FULL, !walk);
    if (idle) {
      while (qh == qn && unit < units) {
        qh = qn = 0;
        if (FIRST) {
          const uint32_t row = (uint32_t)(unit / cpr);
          const uint32_t v0 = (uint32_t)(unit - (uint64_t)row * cpr) * PK_CHUNK;
          qb = row * ld;
          const uint32_t* src = F + qb;
          uint4 w4[2];
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const uint32_t vv = v0 + i * 128 + lane * 4;
            w4[i] = vv < n ? __ldcg(reinterpret_cast<const uint4*>(src + vv)) : make_uint4(n, n, n, n);
          }
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const uint32_t vv = v0 + (i >> 2) * 128 + lane * 4 + (i & 3);
            const uint4 ww = w4[i >> 2];
            const uint32_t w = (i & 3) == 0 ? ww.x : (i & 3) == 1 ? ww.y : (i & 3) == 2 ? ww.z : ww.w;
            const bool cand = vv < n && w != n && w > vv;  // a walk that does not stop at once
            const unsigned m = __ballot_sync(FULL, cand);
            if (cand) q[qn + __popc(m & lt)] = make_uint2(vv, w);
            qn += __popc(m);
          }
        } else {
          const uint32_t i = (uint32_t)unit * 32u + lane;
          uint32_t it = 0, w = n;
          if (i < cnt) {
            it = __ldcg(list + i);
            w = ld_top(F + it) & PW_ID;
          }
          const unsigned m = __ballot_sync(FULL, w != n);
          if (w != n) q[__popc(m & lt)] = make_uint2(it, w);
          qn = __popc(m);
        }
        unit += nw;
        __syncwarp();
      }
      const int r = __popc(idle & lt);
      if (!walk && r < qn - qh) {
        const uint2 cw = q[qh + r];
        if (FIRST) {
          rb = qb;
          v = cw.x;
        } else {
          rb = cw.x / ld * ld;
          v = cw.x - rb;
        }
        x = tort = cw.y;
        lam = pw = 2;
        iters = 0;
        walk = true;
      }
      __syncwarp();
      qh = min(qn, qh + __popc(idle));
      if (!__any_sync(FULL, walk)) break;
    }
    // ---- steps: until a lane is idle and another vertex may be had ----
#pragma unroll 1
    for (int s = 0; s < 4; ++s) {
      bool put = false;
      uint32_t pv = 0;
      if (walk) {
        const uint32_t w = ld_top(F + rb + x);
        const uint32_t y = w & PW_ID;
        if (emit) {
          put = true;
          pv = rb + x;
          ++clen;
          if (y == v) {  // the cycle is listed
            emit = walk = false;
            pops += clen;
            if (p.steps != nullptr) {
              int32_t a;
              int64_t t;
              row_of(p, g0 + rb / ld, &a, &t);
              atomicAdd(p.steps + (p.num_graphs > 0 ? (size_t)p.gid[v] : (size_t)a) * p.tau + (size_t)t,
                        (unsigned long long)clen);
            }
          }
          x = y;
        } else if (!FIRST && (w & act) && x < v) {
          walk = false;
        } else if (y == n || (FIRST && y < v)) {
          walk = false;
        } else if (y == v) {  // v's cycle: go round once more and list it
          emit = true;
          clen = 1;
          put = true;
          pv = rb + v;
          x = ld_top(F + rb + v) & PW_ID;
        } else if (y == tort) {
          walk = false;
        } else {
          x = y;
          if (--lam == 0u) {
            tort = y;
            pw <<= 1;
            lam = pw;
          }
        }
        if (++iters > p.max_iters) {
          atomicOr(p.err, ERR_TIMEOUT);
          walk = emit = false;
        }
      }
      const unsigned m = __ballot_sync(FULL, put);
      if (m) {
        if (ne + __popc(m) > PK_EMIT) {
          uint32_t b = 0;
          if (lane == 0) b = atomicAdd(outcnt, (uint32_t)ne);
          b = __shfl_sync(FULL, b, 0);
          for (int i = lane; i < ne; i += 32) out[b + i] = em[i];
          ne = 0;
          __syncwarp();
        }
        if (put) em[ne + __popc(m & lt)] = pv;
        ne += __popc(m);
        __syncwarp();
      }
    }
  }
  if (ne) {
    uint32_t b = 0;
    if (lane == 0) b = atomicAdd(outcnt, (uint32_t)ne);
    b = __shfl_sync(FULL, b, 0);
    for (int i = lane; i < ne; i += 32) out[b + i] = em[i];
  }
  __syncwarp();
  return pops;
}

template <bool WGT>
__global__ void __launch_bounds__(PK_T, 4) k_pop(PopParams p) {
  __shared__ uint2 sh_q[PK_W][PK_CHUNK];
  __shared__ uint32_t sh_e[PK_W][PK_EMIT];
  const int team = (int)(blockIdx.x / (unsigned)p.ctas), cta = (int)(blockIdx.x % (unsigned)p.ctas);
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const size_t cap = (size_t)p.wrows * p.ld;
  uint32_t* F = p.F + (size_t)team * cap;
  uint32_t* K = p.K + (size_t)team * cap;
  uint32_t* L = p.L + (size_t)team * 2 * cap;
  uint32_t* ctl = p.ctl + team * 32;
  uint32_t* lc = ctl + CTL_COUNT;  // list counts, by round mod 3
  uint32_t gen = 0, pops = 0;
  const int64_t windows = (p.total + p.wrows - 1) / p.wrows;
  bool quit = false;
  for (int64_t win = team; win < windows && !quit; win += p.teams) {
    const int64_t g0 = win * p.wrows;
    const int32_t rows = (int32_t)min((int64_t)p.wrows, p.total - g0);
    pop_draw<WGT>(p, F, g0, rows, cta);
    if (cta == 0 && threadIdx.x == 0) {
      lc[0] = lc[1] = 0u;
    }
    if ((quit = team_sync(ctl, p.ctas, gen, p.err))) break;
    uint32_t cnt = 0;
    for (uint32_t rd = 0;; ++rd) {
      // round rd: the list of round rd in L[rd & 1] (every vertex for rd = 0)
      uint32_t* nxt = L + (size_t)((rd + 1) & 1) * cap;
      if (cta == 0 && threadIdx.x == 0) {
        lc[(rd + 2) % 3] = 0u;  // last read two barriers ago
        if (rd > p.max_iters) atomicOr(p.err, ERR_TIMEOUT);
      }
      if (rd == 0)
        pops += pop_walk<true>(p, F, nullptr, 0u, 0, nxt, lc + 1, g0, rows, cta, sh_q[wid], sh_e[wid]);
      else
        pops += pop_walk<false>(p, F, L + (size_t)(rd & 1) * cap, cnt, (int)(rd & 1), nxt, lc + (rd + 1) % 3, g0, rows,
                                cta, sh_q[wid], sh_e[wid]);
      if ((quit = team_sync(ctl, p.ctas, gen, p.err))) break;
      const uint32_t nc = __ldcg(lc + (rd + 1) % 3);
      if (nc == 0u) break;  // uniform: not written before the next barrier
      pop_redraw(p, F, K, nxt, nc, L + (size_t)(rd & 1) * cap, cnt, (int)((rd + 1) & 1), g0, cta);
      cnt = nc;
      if ((quit = team_sync(ctl, p.ctas, gen, p.err))) break;
    }
    if (quit) break;
    if (p.parents != nullptr) {
      const int64_t len = (int64_t)rows * p.n;
      for (int64_t i = (int64_t)cta * PK_T + threadIdx.x; i < len; i += (int64_t)p.ctas * PK_T) {
        const int64_t r = i / p.n;
        p.parents[(g0 + r) * p.n + (i - r * p.n)] = (int32_t)(F[r * p.ld + (i - r * p.n)] & PW_ID);
      }
    }
    if (p.item_ns != nullptr) {
      const unsigned long long ns = global_ns();
      const int64_t len = (int64_t)rows * p.num_graphs;
      for (int64_t i = (int64_t)cta * PK_T + threadIdx.x; i < len; i += (int64_t)p.ctas * PK_T)
        p.item_ns[(i / rows) * p.tau + g0 + i % rows] = ns;
    }
    if ((quit = team_sync(ctl, p.ctas, gen, p.err))) break;  // the tops are read before they are drawn again
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) pops += __shfl_xor_sync(FULL, pops, o);
  if (lane == 0 && pops) {
    atomicAdd(&p.stats[0], (unsigned long long)pops);
    atomicAdd(&p.stats[1], (unsigned long long)pops);
  }
}

__global__ void k_pop_begin(unsigned long long* t0_ns, unsigned long long* stats, unsigned long long departures) {
  if (t0_ns) *t0_ns = global_ns();
  stats[0] = 0;
  stats[1] = departures;
}

}  // namespace

// Bytes of tops per window and team.  A window's phases end with its longest
// walk, so more rows per window spread that wait: measured on GB300 (4 teams),
// windows of 20 / 40 / 80 / 160 / 400 MB: BA n = 2^20, 1024 trees 36.3 / 28.3 /
// 25.0 / 23.7 / 25.8 ms; grid 1024^2, alpha = 10, 152 trees 81.8 / 58.2 / 45.3 /
// 38.9 / 39.2 ms.  One team instead of four: 31.0 and 67.5 ms at 160 MB.
constexpr int64_t POP_WINDOW = 160ll << 20;

static const void* pop_fn(const fc_graph* g) {
  return g->weighted ? (const void*)k_pop<true> : (const void*)k_pop<false>;
}

fc_status pop_plan(const fc_graph* g, int64_t total, PopPlan* pl) {
  int nsm = 0, per_sm = 0, coop = 0;
  FC_CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, g->device));
  FC_CK(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, g->device));
  FC_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, pop_fn(g), PK_T, 0));
  if (!coop || per_sm < 1) {
    set_error("fc_sample_usts: the device does not support cooperative launches");
    return FC_ECUDA;
  }
  const int64_t ld = ((int64_t)g->n + 3) & ~(int64_t)3;
  const int64_t cap = std::max<int64_t>(1, POP_WINDOW / (ld * 4));
  pl->teams = (int)std::min<int64_t>(per_sm, total);
  // 16 bytes per vertex and row (top, entry count, two lists) within a quarter of the device
  while (pl->teams > 1 && (size_t)pl->teams * ld * 16 > g->device_bytes / 4) --pl->teams;
  pl->wrows = (int32_t)std::max<int64_t>(1, std::min<int64_t>(cap, (total + pl->teams - 1) / pl->teams));
  while (pl->wrows > 1 && (size_t)pl->teams * pl->wrows * ld * 16 > g->device_bytes / 4) pl->wrows = (pl->wrows + 1) / 2;
  // CTAs per team: every SM, fewer when a window is small (a barrier of few CTAs is quicker)
  const int64_t full = (int64_t)nsm * (per_sm / pl->teams);
  const int64_t want = ((int64_t)pl->wrows * g->n + 4 * PK_T - 1) / (4 * PK_T);
  pl->ctas = (int)std::max<int64_t>(1, std::min<int64_t>(full, want));
  pl->bytes = (size_t)pl->teams * pl->wrows * ld * 16 + (size_t)pl->teams * 128;
  return FC_OK;
}

fc_status pop_sample(fc_graph* g, const WParams& w, const PopPlan& pl, void* ws, cudaStream_t st) {
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
  FC_CK(cudaMemsetAsync(p.ctl, 0, (size_t)pl.teams * 128, st));
  k_pop_begin<<<1, 1, 0, st>>>(w.t0_ns, w.stats, (unsigned long long)g->n * (unsigned long long)p.total);
  FC_LAUNCHED();
  void* args[] = {&p};
  FC_CK(cudaLaunchCooperativeKernel(pop_fn(g), dim3((unsigned)(pl.teams * pl.ctas)), dim3(PK_T), args, 0, st));
  FC_LAUNCHED();
  g->last_W = PK_T;
  g->last_regs = 64;
  g->last_grid = pl.teams * pl.ctas;
  g->last_kernel = 5;
  g->last_cluster = 1;
  return FC_OK;
}

}  // namespace fcx
