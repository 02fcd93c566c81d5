// local_move.cu — the local-moving phase (Section 3.2 of the paper).
//
// For every visited vertex i: sum the edge weight from i to each neighbouring
// community (K_{i->c}, self-loop excluded), evaluate the exact gain of moving
// to each of them, and move to the best one if its gain is positive (ties to
// the lowest community id).  The paper's per-thread hashtable becomes, here,
// one table per vertex sized to its degree class:
//
//   bucket 0  degree 1..8       one thread per vertex, table in registers
//   bucket 1  degree 9..32      one thread per vertex, row sorted in registers
//                               (128-bit gains: one warp, 64-slot shared table)
//   bucket 2  degree 33..128    one warp per vertex, 256-slot shared table
//   bucket 3  degree 129..1024  one block per vertex, 2048-slot shared table
//   bucket 4  degree 1025..4096 one block per vertex, 8192-slot shared table
//   bucket 5  degree 4097..12288  one block per vertex, 18432-slot shared table
//   bucket 6  larger degrees    hub: several blocks insert into a global
//                               table of 2*degree slots, one block decides
//
// Synchronous mode (Jacobi): decisions read the state at the start of the
// class and append (vertex, target) to a move list; lm_commit applies the
// list afterwards.  Asynchronous mode (Gauss-Seidel-like): a decision is
// applied at once (memberships stored, totals and sizes updated with
// atomics), so later decisions may see it.  A small graph that one block takes
// (lm_small) is the exception: of two classes and more, a class's moves are
// applied when the class is done, in either mode.
#include <algorithm>
#include <climits>
#include "common.cuh"
#include "engine.h"

namespace gbl {

// --------------------------------------------------------- small helpers

__device__ __forceinline__ unsigned lanemask_lt_lm() {
  unsigned m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// Loads of memberships, community totals and sizes.  LD 0: read-only path
// (nothing writes them while the kernel runs: a synchronous class); 1: plain
// (asynchronous in-place updates, any recent value will do: exactly the
// staleness that mode allows).
template <int LD, typename T>
__device__ __forceinline__ T ld_state(const T* p) {
  if (LD == 0) return __ldg(p);
  return *p;
}
template <bool ASYNC>
__device__ __forceinline__ int32_t ld_memb(const int32_t* p) {
  return ld_state<ASYNC ? 1 : 0>(p);
}
template <bool ASYNC>
__device__ __forceinline__ long long ld_sig(const long long* p) {
  return ld_state<ASYNC ? 1 : 0>(p);
}
template <bool ASYNC>
__device__ __forceinline__ int32_t ld_size(const int32_t* p) {
  return ld_state<ASYNC ? 1 : 0>(p);
}

// Block-level accumulators, flushed once per block.
struct BlockAcc {
  unsigned long long moves, edges, visited, s_lo, s_hi, cands;
  int error;
};

__device__ __forceinline__ void acc_init(BlockAcc& b) {
  if (threadIdx.x == 0) { b.moves = 0; b.edges = 0; b.visited = 0; b.s_lo = 0; b.s_hi = 0; b.cands = 0; b.error = 0; }
}
__device__ __forceinline__ void acc_flush(BlockAcc& b, DevCounters* ctr) {
  if (threadIdx.x == 0) {
    if (b.moves) atomicAdd(&ctr->moves, b.moves);
    if (b.edges) atomicAdd(&ctr->edges, b.edges);
    if (b.visited) atomicAdd(&ctr->visited, b.visited);
    if (b.cands) atomicAdd(&ctr->cands, b.cands);
    u128 s = ((u128)b.s_hi << 64) | (u128)b.s_lo;
    if (s) atomic_add_u128(&ctr->s_lo, &ctr->s_hi, s);
    if (b.error) atomicOr(&ctr->error, b.error);
  }
}

__device__ __forceinline__ u128 warp_sum_u128(u128 v) {
  unsigned long long lo = (unsigned long long)v, hi = (unsigned long long)(v >> 64);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long l2 = __shfl_xor_sync(0xffffffffu, lo, o), h2 = __shfl_xor_sync(0xffffffffu, hi, o);
    const unsigned long long nl = lo + l2;
    hi = hi + h2 + (nl < lo ? 1ull : 0ull);
    lo = nl;
  }
  return ((u128)hi << 64) | (u128)lo;
}

// All 32 lanes of a warp: the moves and gains of the lanes that moved (gv of
// a lane that did not is ignored), summed per graph of a batch and added
// with one atomic per distinct graph, or to the block's accumulator.
template <typename W>
__device__ __forceinline__ void warp_move_totals(const LMArgs<W>& a, BlockAcc& acc, bool moved, int graph, u128 gv) {
  unsigned pend = __ballot_sync(0xffffffffu, moved);
  while (pend) {
    const int leader = __ffs(pend) - 1;
    const int gl = __shfl_sync(0xffffffffu, graph, leader);
    const bool in = moved && (!a.gid || graph == gl);
    const unsigned inm = __ballot_sync(0xffffffffu, in);
    const u128 sum = warp_sum_u128(in ? gv : (u128)0);
    if ((int)(threadIdx.x & 31) == leader) {
      if (a.gid) {
        atomicAdd(a.g_moves + gl, (unsigned long long)__popc(inm));
        atomic_add_u128(a.g_s + 2 * gl, a.g_s + 2 * gl + 1, sum);
      } else {
        atomicAdd(&acc.moves, (unsigned long long)__popc(inm));
        atomic_add_u128(&acc.s_lo, &acc.s_hi, sum);
      }
    }
    pend &= ~inm;
  }
}

// Decide-and-apply for vertex i (called by one thread): guard, then either
// an in-place move (asynchronous) or an entry in the move list (synchronous).
// Returns whether the vertex moves.
// `best` is the best candidate's score, `score_d` the vertex's own; the move
// needs gain = best - score_d > 0.
// sd, szd: Sigma_d and the size of d, loaded with the vertex's row (constant
// within a synchronous class; an asynchronous decision may use any recent
// value).  size_c: the size of c when the caller loaded it with the
// candidates (the guard's test), else -1 and it is loaded here.
// LIST false: a synchronous move is not appended here (the caller does it for
// the whole warp).
template <typename W, bool WIDE, bool ASYNC, int LD = (ASYNC ? 1 : 0), bool LIST = true>
__device__ __forceinline__ bool commit_choice(const LMArgs<W>& a, BlockAcc& acc, int32_t i, int32_t d, long long Ki,
                                              long long sd, int32_t szd, typename Arith<WIDE>::S best, int32_t c,
                                              unsigned long long kid, long long M, int graph,
                                              u128* defer_gain = nullptr, int32_t size_c = -1) {
  if (c < 0) return false;
  typedef typename Arith<WIDE>::S S;
  const S g = best - Arith<WIDE>::score(M, (long long)kid, Ki, sd - Ki);
  if (!(g > 0)) return false;
  if (a.guard && c > d && szd == 1 && (size_c >= 0 ? size_c : ld_state<LD>(a.csize + c)) == 1) return false;
  if (ASYNC) {
    a.memb[i] = c;
    atomicAdd((unsigned long long*)(a.sig + d), (unsigned long long)(-Ki));
    atomicAdd((unsigned long long*)(a.sig + c), (unsigned long long)Ki);
    atomicSub(a.csize + d, 1);
    atomicAdd(a.csize + c, 1);
  } else if (LIST) {
    unsigned long long pos = atomicAdd(a.ctr->nmoves_list + a.odd, 1ull);
    a.moves[pos] = make_int2(i, c);
  }
  u128 gv = Arith<WIDE>::to_u128(g);   // g > 0 here
  if (defer_gain) {   // the caller adds the move and its gain
    *defer_gain = gv;
    return true;
  }
  if (a.gid) {
    atomicAdd(a.g_moves + graph, 1ull);
    atomic_add_u128(a.g_s + 2 * graph, a.g_s + 2 * graph + 1, gv);
  } else {
    atomicAdd(&acc.moves, 1ull);
    atomic_add_u128(&acc.s_lo, &acc.s_hi, gv);
  }
  return true;
}

// The graph of vertex i and its M; false if that graph has stopped
// iterating in this pass.
template <typename W>
__device__ __forceinline__ bool graph_of(const LMArgs<W>& a, int32_t i, long long* M, int* g) {
  if (!a.gid) {
    *M = a.M;
    *g = 0;
    return true;
  }
  const int gg = a.gid[i];
  *g = gg;
  if (!a.g_on[gg]) return false;
  *M = a.Mg[gg];
  return true;
}

// The iteration and its stamp buffers, read once at kernel start.
struct IterView {
  int iter;
  const int32_t* sr;   // read: active in this iteration
  int32_t* sw;         // write: active in the next one
};

template <typename W>
__device__ __forceinline__ IterView iter_view(const LMArgs<W>& a) {
  const int it = *a.d_iter;
  return IterView{it, a.stamps[it & 1], a.stamps[(it + 1) & 1]};
}

// Pruning by pull, while nearly every vertex is active (synchronous).
// A vertex is active when it or a neighbour moved in the iteration before.
// Pushed, every mover rereads its row and stores a stamp per neighbour, twenty
// stores for one vertex and most of them to the same hubs (R-MAT of 4.2M
// vertices: 21 of 117 ms).  Instead a move sets a flag in the mover's own
// membership word, one of two bits above the ids by the iteration's parity; a
// vertex's row is gathered anyway, so it sees its neighbours' flags for nothing,
// and only the few inactive vertices gather for nothing.  The flags are cleared
// at the end of the iteration that read them.  Bound by the gathers of the
// neighbours' words, as before; a run of the R-MAT graph went from 116.8 to
// 100.5 ms, an incremental one of 1M vertices from 13.1 to 11.0, a 4096 x 4096
// road grid from 36.1 to 34.6.
constexpr int32_t kIdMask = 0x3fffffff;
__device__ __forceinline__ int32_t moved_bit(int iter) { return (iter & 1) ? (int32_t)0x80000000 : 0x40000000; }
// A membership word as a community id.
template <bool PULL>
__device__ __forceinline__ int32_t word_id(int32_t w) {
  return PULL ? (w & kIdMask) : w;
}

template <bool PULL = false, typename W>
__device__ __forceinline__ bool is_active(const LMArgs<W>& a, const IterView& iv, int32_t i) {
  return !a.prune || iv.iter == 0 || (PULL && a.pull_check) || iv.sr[i] == iv.iter;
}

// What a warp or block needs of a vertex before its row.
struct VertexRow {
  int32_t i, d;   // the vertex and its community
  int deg;
  int64_t b;      // first entry of its row
  long long Ki;
  int graph;      // set by window_row
  long long M;
};

// A window of 32 list entries first, first + stride, ...: lane l loads entry
// first + l * stride, so one chain of dependent loads (list entry, stamp, row
// bounds, community, degree) serves 32 vertices and inactive vertices cost
// nothing more.  Returns the lanes whose vertex is visited in this iteration.
// A vertex's own community only changes by its own commit, so it may be read
// ahead; its community's total and size are read when its row is.
template <typename W, bool PULL = false>
__device__ __forceinline__ unsigned vertex_window(const LMArgs<W>& a, const IterView& iv,
                                                  const int32_t* __restrict__ verts, int64_t nverts, int64_t first,
                                                  int64_t stride, int lane, VertexRow& r) {
  bool on = false;
  const int64_t at = first + lane * stride;
  r = VertexRow{0, 0, 0, 0, 0, 0, 0};
  if (at < nverts) {
    r.i = verts[at];
    if (is_active<PULL>(a, iv, r.i) && (!a.gid || a.g_on[a.gid[r.i]])) {
      on = true;
      r.b = a.off[r.i];
      r.deg = (int)(a.off[r.i + 1] - r.b);
      r.d = ld_state<1>(a.memb + r.i);
      r.Ki = a.K[r.i];
    }
  }
  return __ballot_sync(0xffffffffu, on);
}

// Lane src's vertex of a window, to every lane.
template <typename W>
__device__ __forceinline__ VertexRow window_row(const LMArgs<W>& a, const VertexRow& r, int src) {
  VertexRow v;
  v.i = __shfl_sync(0xffffffffu, r.i, src);
  v.d = __shfl_sync(0xffffffffu, r.d, src);
  v.deg = __shfl_sync(0xffffffffu, r.deg, src);
  v.b = __shfl_sync(0xffffffffu, r.b, src);
  v.Ki = __shfl_sync(0xffffffffu, r.Ki, src);
  v.graph = 0;
  v.M = a.M;
  if (a.gid) {
    v.graph = a.gid[v.i];
    v.M = a.Mg[v.graph];
  }
  return v;
}

// Pruning marks of a vertex that moved: the vertex and every neighbour are
// active in the next iteration.  The row's columns are loaded together
// before the marks are stored (a load after a store to the stamps would wait
// for it), U at a time per thread; the entries b + lane0, + step, ... are
// this thread's, and the thread with lane0 == 0 marks the vertex itself.
template <int U, typename W>
__device__ __forceinline__ void mark_row(const LMArgs<W>& a, const IterView& iv, int32_t i, int64_t b, int64_t e,
                                         int lane0 = 0, int step = 1, bool self = true) {
  if (self && lane0 == 0) iv.sw[i] = iv.iter + 1;
  for (int64_t x0 = b + lane0; x0 < e; x0 += (int64_t)U * step) {
    int32_t cc[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t x = x0 + (int64_t)u * step;
      cc[u] = x < e ? __ldg(a.col + x) : -1;
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (cc[u] >= 0) iv.sw[cc[u]] = iv.iter + 1;
  }
}

// --------------------------------------------- bucket 0: thread per vertex

// Synchronous moves of a warp's lanes (all 32 call it), appended to the move
// list with one atomic: neighbouring records come from neighbouring vertices,
// so the commit's loads coalesce.
template <typename W>
__device__ __forceinline__ void append_moves(const LMArgs<W>& a, bool moved, int32_t i, int32_t c) {
  const unsigned m = __ballot_sync(0xffffffffu, moved);
  if (!m) return;
  const int leader = __ffs(m) - 1;
  unsigned long long base = 0;
  if ((int)(threadIdx.x & 31) == leader) base = atomicAdd(a.ctr->nmoves_list + a.odd, (unsigned long long)__popc(m));
  base = __shfl_sync(0xffffffffu, base, leader);
  if (moved) a.moves[base + __popc(m & lanemask_lt_lm())] = make_int2(i, c);
}

// Vertex i (on: it is visited) of degree deg <= D by one lane, row at b: the
// row is loaded first and its neighbours' communities gathered with all loads
// in flight; duplicates are then merged in registers.  gv: the gain of a move.
// A synchronous move is left to the caller's append (to: its target).
// *on is cleared when a vertex taken for active (PULL) is not.
template <typename W, bool WIDE, bool ASYNC, bool PULL, int D>
__device__ __forceinline__ bool thread_decide(const LMArgs<W>& a, const IterView& iv, BlockAcc& acc, int32_t i,
                                              int64_t b, int deg, int32_t dw, long long Ki, long long M, int graph,
                                              int32_t* to, u128* gv, unsigned* n_cand, bool* on) {
  const int32_t d = word_id<PULL>(dw);
  typedef typename Arith<WIDE>::S S;
  typedef typename TableVal<WIDE>::T V;
  const long long sd = ld_sig<ASYNC>(a.sig + d);
  const int32_t szd = ld_size<ASYNC>(a.csize + d);
  int32_t cc[D];
  V ww[D];
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const bool v = k < deg;
    cc[k] = v ? a.col[b + k] : i;
    ww[k] = v ? (V)a.wt[b + k] : (V)0;
  }
#pragma unroll
  for (int k = 0; k < D; ++k) cc[k] = cc[k] != i ? ld_memb<ASYNC>(a.memb + cc[k]) : kEmpty;
  if (PULL) {
    int32_t seen = dw;
#pragma unroll
    for (int k = 0; k < D; ++k)
      if (cc[k] != kEmpty) {
        seen |= cc[k];
        cc[k] &= kIdMask;
      }
    if (a.pull_check && !(seen & moved_bit(iv.iter - 1))) {
      *on = false;
      return false;
    }
  }
#pragma unroll
  for (int k = 1; k < D; ++k) {
    bool merged = false;
#pragma unroll
    for (int l = 0; l < k; ++l)
      if (!merged && cc[k] != kEmpty && cc[l] == cc[k]) { ww[l] += ww[k]; merged = true; }
    if (merged) cc[k] = kEmpty;
  }
  V kid = 0;
#pragma unroll
  for (int k = 0; k < D; ++k)
    if (cc[k] == d) kid = ww[k];
  // the candidates' totals, and for a singleton under the guard their
  // sizes too (loaded with the totals instead of after the choice)
  const bool want_size = a.guard && szd == 1;
  long long sg[D];
  int32_t sz[D];
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const bool cand = cc[k] != kEmpty && cc[k] != d;
    sg[k] = cand ? ld_sig<ASYNC>(a.sig + cc[k]) : 0;
    sz[k] = cand && want_size && cc[k] > d ? ld_size<ASYNC>(a.csize + cc[k]) : 0;
  }
  S bg = Arith<WIDE>::lowest();
  int32_t bc = -1, bsz = 0;
  unsigned ncand = 0;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    if (cc[k] != kEmpty && cc[k] != d) {
      ++ncand;
      S g = Arith<WIDE>::score(M, (long long)ww[k], Ki, sg[k]);
      if (better(g, cc[k], bg, bc)) { bg = g; bc = cc[k]; bsz = sz[k]; }
    }
  }
  *n_cand = ncand;
  *to = bc;
  return commit_choice<W, WIDE, ASYNC, (ASYNC ? 1 : 0), false>(a, acc, i, d, Ki, sd, szd, bg, bc, kid, M, graph, gv,
                                                              bsz);
}

// Up to 32 visited vertices, a lane each (i < 0: none); all 32 lanes call it.
// A warp whose rows all have at most four entries (a road grid's nearly all
// do) takes the instance that compares six pairs instead of 28.  Whole warps
// sum their counters, moves and gains over the warp: per-lane atomics on the
// block's counters serialise (measured: a third of the kernel's time).
template <typename W, bool WIDE, bool ASYNC, bool PULL = false>
__device__ __forceinline__ void thread_vertices(const LMArgs<W>& a, const IterView& iv, BlockAcc& acc, int32_t i) {
  int64_t b = 0;
  int deg = 0, graph = 0;
  int32_t d = 0, to = -1;
  long long Ki = 0, M = 0;
  if (i >= 0) {
    b = a.off[i];
    deg = (int)(a.off[i + 1] - b);
    d = a.memb[i];
    Ki = a.K[i];
    M = a.M;
    if (a.gid) {
      graph = a.gid[i];
      M = a.Mg[graph];
    }
  }
  bool moved = false, on = i >= 0;
  u128 gv = 0;
  unsigned n_cand = 0;
  const unsigned longest = __reduce_max_sync(0xffffffffu, (unsigned)deg);
  if (longest <= 4) {
    if (i >= 0)
      moved = thread_decide<W, WIDE, ASYNC, PULL, 4>(a, iv, acc, i, b, deg, d, Ki, M, graph, &to, &gv, &n_cand, &on);
  } else {
    if (i >= 0)
      moved = thread_decide<W, WIDE, ASYNC, PULL, 8>(a, iv, acc, i, b, deg, d, Ki, M, graph, &to, &gv, &n_cand, &on);
  }
  if (moved && a.prune && !(PULL && a.pull_mark)) mark_row<8>(a, iv, i, b, b + deg);
  if (!ASYNC) append_moves(a, moved, i, to);
  const unsigned n_edges = __reduce_add_sync(0xffffffffu, PULL && !on ? 0u : (unsigned)deg);
  const unsigned n_visited = (unsigned)__popc(__ballot_sync(0xffffffffu, on));
  n_cand = __reduce_add_sync(0xffffffffu, n_cand);
  if ((threadIdx.x & 31) == 0 && n_visited) {
    atomicAdd(&acc.edges, (unsigned long long)n_edges);
    atomicAdd(&acc.visited, (unsigned long long)n_visited);
    atomicAdd(&acc.cands, (unsigned long long)n_cand);
  }
  warp_move_totals(a, acc, moved, graph, gv);
}

// Lane l takes list entry base + l (none past nverts or inactive).
template <typename W, bool WIDE, bool ASYNC>
__device__ __forceinline__ void thread_vertex(const LMArgs<W>& a, const IterView& iv, BlockAcc& acc,
                                              const int32_t* __restrict__ verts, int64_t nverts, int64_t vi) {
  int32_t i = -1;
  if (vi < nverts) {
    i = verts[vi];
    if (!is_active(a, iv, i) || (a.gid && !a.g_on[a.gid[i]])) i = -1;
  }
  if (__any_sync(0xffffffffu, i >= 0)) thread_vertices<W, WIDE, ASYNC>(a, iv, acc, i);
}

// The warp walks its list entries 32 at a time and queues the visited ones in
// shared memory until 32 are there: with pruning most lanes of a warp would
// otherwise idle through the others' rows.
template <typename W, bool WIDE, bool ASYNC, bool PULL>
__global__ void __launch_bounds__(256, 3) lm_thread(LMArgs<W> a, const int32_t* __restrict__ list,
    const int64_t* __restrict__ ko) {
  const IterView iv = iter_view(a);
  if (iv.iter < 0) return;
  const int32_t* __restrict__ verts = list + ko[0];
  const int nverts = (int)(ko[1] - ko[0]);
  __shared__ BlockAcc acc;
  __shared__ int32_t queue[8][2 * kWarp];
  acc_init(acc);
  __syncthreads();
  const int lane = threadIdx.x & 31;
  int32_t* q = queue[threadIdx.x >> 5];
  int have = 0;
  for (int64_t base = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); base < nverts;
       base += (int64_t)gridDim.x * blockDim.x) {
    int32_t i = -1;
    if (base + lane < nverts) {
      i = verts[base + lane];
      if (!is_active<PULL>(a, iv, i) || (a.gid && !a.g_on[a.gid[i]])) i = -1;
    }
    const unsigned on = __ballot_sync(0xffffffffu, i >= 0);
    if (have == 0 && on == 0xffffffffu) {   // nothing to gather
      thread_vertices<W, WIDE, ASYNC, PULL>(a, iv, acc, i);
      continue;
    }
    if (i >= 0) q[have + __popc(on & lanemask_lt_lm())] = i;
    have += __popc(on);
    __syncwarp();
    if (have >= kWarp) {
      const int32_t j = q[lane];
      const int32_t rest = q[kWarp + lane];
      __syncwarp();
      q[lane] = rest;
      have -= kWarp;
      __syncwarp();
      thread_vertices<W, WIDE, ASYNC, PULL>(a, iv, acc, j);
    }
  }
  if (have > 0) thread_vertices<W, WIDE, ASYNC, PULL>(a, iv, acc, lane < have ? q[lane] : -1);
  __syncthreads();
  acc_flush(acc, a.ctr);
}

// --------------------- bucket 1, narrow arithmetic: thread per vertex, sorted

// A vertex of degree <= D by one lane: its row is loaded and the neighbours'
// communities gathered with all loads in flight, the (community, weight)
// pairs sorted by community with a bitonic network in registers (static
// indices), each run of one community summed into its first position, and the
// runs' totals gathered in two halves (bounded registers).  Same decisions as
// the warp kernel it replaces for narrow sums (K_{i->c} < 2^31).  All 32
// lanes call it.
template <typename W, bool ASYNC, bool PULL, int D>
__device__ __forceinline__ void thread_vertex_sorted(const LMArgs<W>& a, const IterView& iv, BlockAcc& acc,
                                                     const int32_t* __restrict__ verts, int64_t nverts, int64_t vi) {
  typedef typename Arith<false>::S S;
  static_assert((D & (D - 1)) == 0 && D <= 32, "power-of-two network of at most 32");
  constexpr int32_t kPast = 0x7fffffff;   // sorts after every community id
  constexpr int H = D / 2;
  bool moved = false;
  u128 gv = 0;
  int graph = 0;
  int32_t vert = 0, to = -1;
  unsigned n_edges = 0, n_visited = 0, n_cand = 0;
  do {
    if (vi >= nverts) break;
    const int32_t i = verts[vi];
    const int64_t b = a.off[i], e = a.off[i + 1];
    const int32_t dw = a.memb[i], d = word_id<PULL>(dw);
    const long long Ki = a.K[i];
    if (!is_active<PULL>(a, iv, i)) break;
    long long M;
    if (!graph_of(a, i, &M, &graph)) break;
    const long long sd = ld_sig<ASYNC>(a.sig + d);
    const int32_t szd = ld_size<ASYNC>(a.csize + d);
    int32_t k[D];
    unsigned w[D];
#pragma unroll
    for (int j = 0; j < D; ++j) {
      const bool v = b + j < e;
      k[j] = v ? a.col[b + j] : i;
      w[j] = v ? (unsigned)a.wt[b + j] : 0u;
    }
#pragma unroll
    for (int j = 0; j < D; ++j) {
      const bool other = k[j] != i;   // a self-loop adds to no K_{i->c}
      k[j] = other ? ld_memb<ASYNC>(a.memb + k[j]) : kPast;
      if (!other) w[j] = 0u;
    }
    if (PULL) {
      int32_t seen = dw;
#pragma unroll
      for (int j = 0; j < D; ++j)
        if (k[j] != kPast) {
          seen |= k[j];
          k[j] &= kIdMask;
        }
      if (a.pull_check && !(seen & moved_bit(iv.iter - 1))) break;
    }
#pragma unroll
    for (int kk = 2; kk <= D; kk <<= 1) {
#pragma unroll
      for (int jj = kk >> 1; jj > 0; jj >>= 1) {
#pragma unroll
        for (int x = 0; x < D; ++x) {
          const int y = x ^ jj;
          if (y > x) {
            const bool up = (x & kk) == 0;
            if ((k[x] > k[y]) == up) {
              const int32_t tk = k[x]; k[x] = k[y]; k[y] = tk;
              const unsigned tw = w[x]; w[x] = w[y]; w[y] = tw;
            }
          }
        }
      }
    }
    // run heads (first position of each community) carry the run's sum
    unsigned heads = 0u, run = 0u;
#pragma unroll
    for (int j = D - 1; j >= 0; --j) {
      run += w[j];
      if (k[j] != kPast && (j == 0 || k[j] != k[j - 1])) {
        heads |= 1u << j;
        w[j] = run;
        run = 0u;
      }
    }
    unsigned long long kid = 0;
#pragma unroll
    for (int j = 0; j < D; ++j)
      if (((heads >> j) & 1u) && k[j] == d) kid = w[j];
    const bool want_size = a.guard && szd == 1;
    S bg = Arith<false>::lowest();
    int32_t bc = -1, bsz = 0;
    unsigned ncand = 0;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      long long sg[H];
      bool one[H];
#pragma unroll
      for (int t = 0; t < H; ++t) {
        const int j = half * H + t;
        const bool cand = ((heads >> j) & 1u) && k[j] != d;
        sg[t] = cand ? ld_sig<ASYNC>(a.sig + k[j]) : 0;
        one[t] = cand && want_size && k[j] > d && ld_size<ASYNC>(a.csize + k[j]) == 1;
      }
#pragma unroll
      for (int t = 0; t < H; ++t) {
        const int j = half * H + t;
        if (((heads >> j) & 1u) && k[j] != d) {
          ++ncand;
          const S g = Arith<false>::score(M, (long long)w[j], Ki, sg[t]);
          if (better(g, k[j], bg, bc)) { bg = g; bc = k[j]; bsz = one[t] ? 1 : 0; }
        }
      }
    }
    n_cand = ncand;
    n_edges = (unsigned)(e - b);
    n_visited = 1;
    moved = commit_choice<W, false, ASYNC, (ASYNC ? 1 : 0), false>(a, acc, i, d, Ki, sd, szd, bg, bc, kid, M, graph,
                                                                   &gv, bsz);
    vert = i;
    to = bc;
    if (moved && a.prune && !(PULL && a.pull_mark)) mark_row<8>(a, iv, i, b, e);
  } while (false);
  if (!ASYNC) append_moves(a, moved, vert, to);
  n_edges = __reduce_add_sync(0xffffffffu, n_edges);
  n_visited = __reduce_add_sync(0xffffffffu, n_visited);
  n_cand = __reduce_add_sync(0xffffffffu, n_cand);
  if ((threadIdx.x & 31) == 0 && n_visited) {
    atomicAdd(&acc.edges, (unsigned long long)n_edges);
    atomicAdd(&acc.visited, (unsigned long long)n_visited);
    atomicAdd(&acc.cands, (unsigned long long)n_cand);
  }
  warp_move_totals(a, acc, moved, graph, gv);
}

template <typename W, bool ASYNC, bool PULL, int D>
__global__ void __launch_bounds__(128) lm_thread_sorted(LMArgs<W> a, const int32_t* __restrict__ list,
    const int64_t* __restrict__ ko) {
  const IterView iv = iter_view(a);
  if (iv.iter < 0) return;
  const int32_t* __restrict__ verts = list + ko[0];
  const int nverts = (int)(ko[1] - ko[0]);
  __shared__ BlockAcc acc;
  acc_init(acc);
  __syncthreads();
  for (int base = blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < nverts; base += gridDim.x * blockDim.x)
    thread_vertex_sorted<W, ASYNC, PULL, D>(a, iv, acc, verts, nverts, base + (int)(threadIdx.x & 31));
  __syncthreads();
  acc_flush(acc, a.ctr);
}

// ------------------------------------------ buckets 1-2: warp per vertex

// Tallies a warp keeps in registers while it walks its vertices, added to the
// block's accumulator once at the end (all 32 lanes call add).
struct WarpTally {
  unsigned long long edges = 0;
  unsigned visited = 0, cands = 0;   // per thread, of one launch
  __device__ __forceinline__ void add(BlockAcc& acc) {
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) edges += __shfl_xor_sync(0xffffffffu, edges, m);
    unsigned long long c = cands;
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) c += __shfl_xor_sync(0xffffffffu, c, m);
    visited = __reduce_add_sync(0xffffffffu, visited);
    if ((threadIdx.x & 31) == 0) {
      if (edges) atomicAdd(&acc.edges, edges);
      if (visited) atomicAdd(&acc.visited, (unsigned long long)visited);
      if (c) atomicAdd(&acc.cands, c);
    }
  }
};

// The U entries of row v that this thread holds (entry u * step + lane0),
// their communities gathered with all loads in flight; kEmpty for none and
// for a self-loop.  Rounds from nu on hold nothing for any lane of the warp.
// Row entries are read once an iteration: kept out of L1, which is left to the
// gathered memberships and totals (R-MAT of 4.2M vertices 101.1 -> 99.3 ms a run,
// 1M vertices with four classes 11.4 -> 11.2, asynchronous sweep 146 -> 143).
__device__ __forceinline__ int32_t ld_row(const int32_t* p) {
  int32_t v;
  asm("ld.global.nc.L1::no_allocate.b32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ int64_t ld_row(const int64_t* p) {
  int64_t v;
  asm("ld.global.nc.L1::no_allocate.b64 %0, [%1];" : "=l"(v) : "l"(p));
  return v;
}

// PULL: returns the flags of the neighbours' words, or-ed.
template <int U, int LD, bool PULL = false, typename W, typename V>
__device__ __forceinline__ int32_t row_communities(const LMArgs<W>& a, const VertexRow& v, int lane0, int step, int nu,
                                                   int32_t (&cc)[U], V (&ww)[U]) {
  const int32_t* __restrict__ col = a.col + v.b;
  const W* __restrict__ wt = a.wt + v.b;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    cc[u] = v.i;
    ww[u] = 0;
    if (u < nu) {
      const int x = u * step + lane0;
      if (x < v.deg) {
        cc[u] = ld_row(col + x);
        ww[u] = (V)ld_row(wt + x);
      }
    }
  }
#pragma unroll
  for (int u = 0; u < U; ++u) cc[u] = u < nu && cc[u] != v.i ? ld_state<LD>(a.memb + cc[u]) : kEmpty;
  int32_t seen = 0;
  if (PULL) {
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (cc[u] != kEmpty) {
        seen |= cc[u];
        cc[u] &= kIdMask;
      }
  }
  return seen;
}

// One vertex of degree <= U * 32 by one warp: its neighbour communities summed
// in the warp's shared table (CAP slots, left empty again), the best score
// against its own community's, the move committed and its neighbours marked.
// The lane whose entry claims a slot keeps the community and the slot in
// registers: it asks for the community's total at once, and after the sums
// are complete it alone evaluates and clears the slot, so nothing scans the
// table.  SIZES: a singleton under the guard loads its candidates' sizes with
// their totals (one dependent load less before the decision; off where the
// registers would spill).
// Returns whether the vertex was active (PULL: known only here).
template <typename W, bool WIDE, bool ASYNC, int CAP, int U, int LD, bool SIZES, bool PULL = false>
__device__ __forceinline__ bool warp_vertex(const LMArgs<W>& a, const IterView& iv, BlockAcc& acc, int32_t* keys,
                                            typename TableVal<WIDE>::T* vals, const VertexRow& v, int lane, bool& ok,
                                            unsigned& cands) {
  typedef typename Arith<WIDE>::S S;
  typedef typename TableVal<WIDE>::T V;
  const int32_t d = word_id<PULL>(v.d);
  const long long sd = ld_state<LD>(a.sig + d);
  const int32_t szd = ld_state<LD>(a.csize + d);
  // rounds of 32 entries that hold at least one (the rest are skipped)
  const int nu = (v.deg + kWarp - 1) / kWarp;
  int32_t cc[U];
  V ww[U];
  int hs[U];
  const int32_t seen = row_communities<U, LD, PULL>(a, v, lane, kWarp, nu, cc, ww);
  if (PULL && a.pull_check && !__any_sync(0xffffffffu, ((seen | v.d) & moved_bit(iv.iter - 1)) != 0)) return false;
  const unsigned fresh = table_add_row<CAP, U, V>(keys, vals, cc, ww, nu, hs, &ok);
  // one lane's reading for the whole warp: it decides which reduction below the
  // lanes take together, and an asynchronous size may change between two loads
  const bool want_size = __shfl_sync(0xffffffffu, (int)(SIZES && a.guard && szd == 1), 0) != 0;
  long long sg[U];
  bool one[U];   // the candidate is a singleton (asked only for the guard)
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const bool cand = ((fresh >> u) & 1u) && cc[u] != d;
    sg[u] = cand ? ld_state<LD>(a.sig + cc[u]) : 0;
    one[u] = cand && want_size && cc[u] > d && ld_state<LD>(a.csize + cc[u]) == 1;
  }
  __syncwarp();   // the sums are complete
  V kid = 0;
  S bg = Arith<WIDE>::lowest();
  int32_t bc = -1, bsz = 0;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    if (!((fresh >> u) & 1u)) continue;
    const V sum = vals[hs[u]];
    if (cc[u] != d) {
      ++cands;
      const S g = Arith<WIDE>::score(v.M, (long long)sum, v.Ki, sg[u]);
      if (better(g, cc[u], bg, bc)) { bg = g; bc = cc[u]; bsz = one[u] ? 1 : 0; }
    } else {
      kid = sum;
    }
    keys[hs[u]] = kEmpty;
    vals[hs[u]] = 0;
  }
  if (want_size) warp_argmax_carry(bg, bc, bsz);
  else warp_argmax(bg, bc);
  {
    const unsigned has = __ballot_sync(0xffffffffu, kid != 0);
    kid = has ? __shfl_sync(0xffffffffu, kid, __ffs(has) - 1) : (V)0;
  }
  bool moved = false;
  if (lane == 0)
    moved = commit_choice<W, WIDE, ASYNC, LD>(a, acc, v.i, d, v.Ki, sd, szd, bg, bc, kid, v.M, v.graph, nullptr,
                                              want_size ? bsz : -1);
  moved = __shfl_sync(0xffffffffu, moved, 0);
  if (moved && a.prune && !(PULL && a.pull_mark)) mark_row<U>(a, iv, v.i, v.b, v.b + v.deg, lane, kWarp);
  return true;
}

// U entries per lane cover the bucket's largest degree: the row is loaded and
// gathered before any insert, so its memory latencies overlap.
template <typename W, bool WIDE, bool ASYNC, bool PULL, int CAP, int U>
__global__ void __launch_bounds__(256, 4) lm_warp(LMArgs<W> a, const int32_t* __restrict__ list,
    const int64_t* __restrict__ ko) {
  const IterView iv = iter_view(a);
  if (iv.iter < 0) return;
  const int32_t* __restrict__ verts = list + ko[0];
  const int nverts = (int)(ko[1] - ko[0]);
  typedef typename TableVal<WIDE>::T V;
  constexpr int WPB = 8;
  __shared__ int32_t skeys[WPB][CAP];
  __shared__ V svals[WPB][CAP];
  __shared__ BlockAcc acc;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  int32_t* keys = skeys[wib];
  V* vals = svals[wib];
  acc_init(acc);
  for (int t = lane; t < CAP; t += kWarp) { keys[t] = kEmpty; vals[t] = 0; }
  __syncthreads();
  bool ok = true;
  WarpTally tally;
  const int64_t stride = (int64_t)gridDim.x * WPB;
  for (int64_t w0 = (int64_t)blockIdx.x * WPB + wib; w0 < nverts; w0 += kWarp * stride) {
    VertexRow r;
    unsigned live = vertex_window<W, PULL>(a, iv, verts, nverts, w0, stride, lane, r);
    if (!(PULL && a.pull_check) && ((live >> lane) & 1u)) {
      tally.edges += (unsigned)r.deg;
      ++tally.visited;
    }
    for (; live; live &= live - 1) {
      const VertexRow v = window_row(a, r, __ffs(live) - 1);
      const bool on = warp_vertex<W, WIDE, ASYNC, CAP, U, (ASYNC ? 1 : 0), false, PULL>(
          a, iv, acc, keys, vals, v, lane, ok, tally.cands);
      if (PULL && a.pull_check && on && lane == 0) {
        tally.edges += (unsigned)v.deg;
        ++tally.visited;
      }
      __syncwarp();
    }
  }
  tally.add(acc);
  if (!__all_sync(0xffffffffu, ok) && lane == 0) atomicOr(&acc.error, kErrProbe);
  __syncthreads();
  acc_flush(acc, a.ctr);
}

// ----------------------------- small pass graphs: one launch per class
//
// When no vertex of the pass graph has degree above 128 and the graph is
// small, the launches of a class are few microseconds of work each: one
// kernel then takes the whole class instead of one kernel per bucket on
// forked streams: a lane per vertex of bucket 0 (as lm_thread), a warp per
// vertex of buckets 1-2 (as lm_warp, 256-slot tables).  ko = the bucket
// offsets of the class lists (device).
template <typename W, bool WIDE, bool ASYNC>
__global__ void __launch_bounds__(256, 3) lm_class(LMArgs<W> a, const int32_t* __restrict__ list,
                                                   const int64_t* __restrict__ ko, int P, int ch) {
  const IterView iv = iter_view(a);
  if (iv.iter < 0) return;
  typedef typename TableVal<WIDE>::T V;
  constexpr int WPB = 8, CAP = 256, U = 4;
  __shared__ int32_t skeys[WPB][CAP];
  __shared__ V svals[WPB][CAP];
  __shared__ BlockAcc acc;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  int32_t* keys = skeys[wib];
  V* vals = svals[wib];
  acc_init(acc);
  for (int t = lane; t < CAP; t += kWarp) { keys[t] = kEmpty; vals[t] = 0; }
  __syncthreads();
  bool ok = true;
  WarpTally tally;
  const int64_t r0 = ko[ch], n0 = ko[ch + 1] - r0;
  const int64_t r1 = ko[P + ch], n1 = ko[P + ch + 1] - r1;
  const int64_t r2 = ko[2 * P + ch], n2 = ko[2 * P + ch + 1] - r2;
  // work items of a warp: 32 degree-<=8 vertices (a lane each, as the thread
  // kernel), then one vertex of degree 9-128 each
  const int64_t m0 = (n0 + kWarp - 1) / kWarp;
  const int64_t tot = m0 + n1 + n2;
  for (int64_t t = (int64_t)blockIdx.x * WPB + wib; t < tot; t += (int64_t)gridDim.x * WPB) {
    if (t < m0) {
      thread_vertex<W, WIDE, ASYNC>(a, iv, acc, list + r0, n0, t * kWarp + lane);
      continue;
    }
    const int64_t u = t - m0;
    const int64_t idx = u < n1 ? r1 + u : r2 + (u - n1);
    VertexRow r;
    if (!vertex_window<W>(a, iv, list + idx, 1, 0, 1, lane, r)) continue;
    if (lane == 0) {
      tally.edges += (unsigned)r.deg;
      ++tally.visited;
    }
    const VertexRow v = window_row(a, r, 0);
    warp_vertex<W, WIDE, ASYNC, CAP, U, (ASYNC ? 1 : 0), !WIDE>(a, iv, acc, keys, vals, v, lane, ok, tally.cands);
    __syncwarp();
  }
  tally.add(acc);
  if (!__all_sync(0xffffffffu, ok) && lane == 0) atomicOr(&acc.error, kErrProbe);
  __syncthreads();
  acc_flush(acc, a.ctr);
}

// ------------------------- small graphs: one block per graph, whole phase
//
// A graph of few thousand vertices leaves most of the chip idle whatever the
// mapping, and a launch per class (5-7 us each, 8 to 32 classes an iteration)
// costs more than its work.  One block then runs every iteration of the phase:
// memberships, totals, sizes and activity bits live in shared memory, a class
// ends at a block barrier, and the iteration's stop test is taken here, on the
// same exact sums and roundings as on the host.  The graphs of a batch run
// side by side, each its own number of iterations.  The classes are those of
// the kernels above.  A class's moves are committed when it is done, in both
// modes, so the results do not vary from run to run.  (An asynchronous graph of
// one class, where that would be the synchronous schedule, takes the launches.)
// Asynchronous Q against the oracle's, means over 12 graphs and 4 runs, here /
// launches: hub-and-spoke of 6,000 vertices, 2 classes -0.0007 / -0.0294, 4
// +0.0004 / -0.0014, 8 +0.0008 / -0.0003; planted partition of 6,000, 2 -0.0013 /
// -0.0014, 8 -0.0001 / -0.0001; grid of 6,400, 4 -0.0004 / -0.0005; R-MAT of
// 4,096, 8 -0.0009 / -0.0004; with 32 classes all within 0.0005 of each other.
// Committing at once let a few decisions see others' moves: 600 vertices in 12
// blocks ended 0.02 lower in Q on average.  A vertex of degree <= 8 takes a
// lane, a larger one a warp.  With at most kTinyVerts vertices every warp has an
// array of sums indexed by community; with more, a table of 256 slots for
// degrees up to 128, and the block together takes larger ones, its warps'
// values forming one such array.

// Vertices of degree above 128 that a graph within the entry limit can hold.
constexpr int kSmallLong = (int)(kSmallEntries / 129) + 1;

// One vertex's best candidate so far.
struct SmallBest {
  long long g;
  int32_t c;
};

template <typename W, int NMAX, int THREADS>
struct SmallGraph {
  static constexpr int NW = THREADS / kWarp;
  static constexpr bool kDense = NMAX <= kTinyVerts;   // sums indexed by community for every warp
  static constexpr int CAP = kDense ? NMAX : 256;      // values of a warp (kDense) or slots of its table
  static constexpr uint16_t kNone = 0xffff;  // no target
  static_assert(NW * CAP >= NMAX, "the values of all tables are one array indexed by community");
  // dynamic shared memory
  long long* sig;      // NMAX
  int32_t* size;       // NMAX
  int32_t* keys;       // NW * CAP, empty between vertices (not with kDense)
  unsigned* vals;      // NW * CAP, zero between vertices
  unsigned* act;       // 2 * NMAX / 32: active in this / the next iteration
  uint16_t* memb;      // NMAX
  uint16_t* list;      // NMAX: vertices with entries by class
  uint16_t* to;        // NMAX: targets of the class's moves
  static constexpr size_t kBytes = (size_t)NMAX * (8 + 4 + 3 * 2) + (size_t)NW * CAP * (kDense ? 4 : 8) + 2 * NMAX / 8;

  __device__ __forceinline__ explicit SmallGraph(void* mem) {
    sig = (long long*)mem;
    size = (int32_t*)(sig + NMAX);
    keys = size + NMAX;
    vals = (unsigned*)(kDense ? keys : keys + NW * CAP);
    act = vals + NW * CAP;
    memb = (uint16_t*)(act + 2 * NMAX / 32);
    list = memb + NMAX;
    to = list + NMAX;
  }
  __device__ __forceinline__ void mark(unsigned* next, int v) const {
    const unsigned bit = 1u << (v & 31);
    if (!(next[v >> 5] & bit)) atomicOr(next + (v >> 5), bit);
  }
  // The gain of moving to the best candidate if the move is taken, else 0.
  __device__ __forceinline__ long long gain(const SmallBest& best, int d, long long Ki, long long M, unsigned kid,
                                            int guard) const {
    if (best.c < 0) return 0;
    const long long g = best.g - Arith<false>::score(M, (long long)kid, Ki, sig[d] - Ki);
    if (g <= 0) return 0;
    if (guard && best.c > d && size[d] == 1 && size[best.c] == 1) return 0;
    return g;
  }
};

template <typename W, int NMAX, int THREADS>
__global__ void __launch_bounds__(THREADS, THREADS == 256 ? 4 : 1) lm_small(LMArgs<W> a, SmallArgs sa) {
  typedef SmallGraph<W, NMAX, THREADS> SG;
  constexpr int NW = SG::NW;
  extern __shared__ unsigned long long sdyn[];
  const SG s(sdyn);
  __shared__ int s_start[66], s_fill[64];
  __shared__ int s_stop, s_moved, s_nlong;
  __shared__ uint16_t s_long[SG::kDense ? 1 : kSmallLong];
  __shared__ unsigned s_kid;
  __shared__ long long r_g[NW];
  __shared__ int32_t r_c[NW];
  __shared__ unsigned long long r_lo[NW], r_hi[NW], r_moves[NW];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const bool single = sa.vo == nullptr;
  const int64_t g = single ? 0 : sa.ids[blockIdx.x];
  const int64_t v0 = single ? 0 : sa.vo[g];
  const int64_t ng = (single ? sa.n : sa.vo[g + 1]) - v0;
  const int64_t nnz = a.off[v0 + ng] - a.off[v0];
  auto rec = [&](int w) -> unsigned long long& { return sa.rec[w * sa.graphs + g]; };
  const int cat = single ? sa.cs.single_cat : sa.gcat[g];
  const int P = cat == kCatSmall ? sa.cs.Ps : cat == kCatSparse ? sa.cs.Pl : sa.cs.Pb;
  const int mode = cat == kCatSmall ? sa.cs.mode_s : sa.cs.mode_b;
  const long long M = single ? a.M : a.Mg[g];
  // 64-bit gains and 32-bit sums must hold every vertex (as for the buckets)
  const long long klimit = M < (1ll << 31) ? M : (long long)((1ull << 61) / (unsigned long long)M);
  int unfit = ng > NMAX || nnz > kSmallEntries;
  if (!unfit)
    for (int v = tid; v < ng; v += THREADS) unfit |= a.K[v0 + v] > klimit;
  if (__syncthreads_or(unfit)) {
    if (tid == 0) rec(0) = kSmallNot;
    return;
  }
  const int n = (int)ng;
  const int64_t* __restrict__ off = a.off + v0;
  for (int v = tid; v < n; v += THREADS) {
    s.memb[v] = (uint16_t)(a.memb[v0 + v] - v0);
    s.sig[v] = a.sig[v0 + v];
    s.size[v] = a.csize[v0 + v];
    s.to[v] = SG::kNone;
  }
  for (int t = tid; t < NW * SG::CAP; t += THREADS) {
    if (!SG::kDense) s.keys[t] = kEmpty;
    s.vals[t] = 0;
  }
  for (int t = tid; t < 2 * NMAX / 32; t += THREADS) s.act[t] = 0;
  if (tid == 0) s_nlong = 0;
  const double MM = u128_to_double((u128)M * (u128)M);
  int32_t* keys = s.keys + wid * SG::CAP;
  unsigned* vals = s.vals + wid * SG::CAP;
  unsigned long long edges = 0;
  unsigned visited = 0, cands = 0;
  bool ok = true;
  int it = 0;
  for (; it < sa.max_iterations; ++it) {
    __syncthreads();
    if (it == 0 || mode == 1) {   // the class lists of this iteration
      for (int c = tid; c < P; c += THREADS) s_fill[c] = 0;
      __syncthreads();
      for (int v = tid; v < n; v += THREADS)
        if (off[v + 1] > off[v])
          atomicAdd(&s_fill[P > 1 ? vertex_class(v0 + v, single ? nullptr : a.gid, sa.vo, sa.gcat, sa.cs, it) : 0], 1);
      __syncthreads();
      if (tid == 0) {
        int sum = 0;
        for (int c = 0; c < P; ++c) {
          const int k = s_fill[c];
          s_start[c] = s_fill[c] = sum;
          sum += k;
        }
        s_start[P] = sum;
      }
      __syncthreads();
      for (int v = tid; v < n; v += THREADS)
        if (off[v + 1] > off[v])
          s.list[atomicAdd(
              &s_fill[P > 1 ? vertex_class(v0 + v, single ? nullptr : a.gid, sa.vo, sa.gcat, sa.cs, it) : 0], 1)] =
              (uint16_t)v;
    }
    const unsigned* cur = s.act + (it & 1) * (NMAX / 32);
    unsigned* next = s.act + ((it + 1) & 1) * (NMAX / 32);
    for (int t = tid; t < NMAX / 32; t += THREADS) next[t] = 0;
    __syncthreads();
    unsigned moves = 0;
    u128 S = 0;
    for (int ch = 0; ch < P; ++ch) {
      const int l0 = s_start[ch], m = s_start[ch + 1] - l0;
      if (m == 0) continue;   // uniform
      // warp w takes entries w, w + NW, ...: 32 of them at a time, a lane each
      for (int j0 = wid; j0 < m; j0 += kWarp * NW) {
        const int j = j0 + lane * NW;
        int v = -1, deg = 0, d = 0;
        int64_t b = 0;
        long long Ki = 0;
        if (j < m) {
          v = s.list[l0 + j];
          if (a.prune && it > 0 && !((cur[v >> 5] >> (v & 31)) & 1u)) v = -1;
        }
        if (v >= 0) {
          b = off[v];
          deg = (int)(off[v + 1] - b);
          Ki = a.K[v0 + v];
          d = s.memb[v];
          edges += (unsigned)deg;
          ++visited;
        }
        if (v >= 0 && deg <= 8) {   // the lane alone
          int cl[8], cc[8];
          unsigned ww[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            cl[k] = k < deg ? (int)(__ldg(a.col + b + k) - v0) : v;
            ww[k] = k < deg ? (unsigned)__ldg(a.wt + b + k) : 0u;
          }
#pragma unroll
          for (int k = 0; k < 8; ++k) cc[k] = cl[k] != v ? (int)s.memb[cl[k]] : kEmpty;
#pragma unroll
          for (int k = 1; k < 8; ++k) {
            bool merged = false;
#pragma unroll
            for (int l = 0; l < k; ++l)
              if (!merged && cc[k] != kEmpty && cc[l] == cc[k]) { ww[l] += ww[k]; merged = true; }
            if (merged) cc[k] = kEmpty;
          }
          unsigned kid = 0;
          SmallBest best{Arith<false>::lowest(), -1};
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            if (cc[k] == kEmpty) continue;
            if (cc[k] == d) {
              kid = ww[k];
            } else {
              ++cands;
              const long long sc =
                  Arith<false>::score(M, (long long)ww[k], Ki, s.sig[cc[k]]);
              if (better(sc, cc[k], best.g, best.c)) best = SmallBest{sc, cc[k]};
            }
          }
          const long long gn = s.gain(best, d, Ki, M, kid, a.guard);
          if (gn) {
            s.to[v] = (uint16_t)best.c;
            ++moves;
            S += (u128)(unsigned long long)gn;
            if (a.prune) {
              s.mark(next, v);
#pragma unroll
              for (int k = 0; k < 8; ++k) s.mark(next, cl[k]);   // cl = v past the row
            }
          }
        }
        for (unsigned big = __ballot_sync(0xffffffffu, v >= 0 && deg > 8); big; big &= big - 1) {
          const int src = __ffs(big) - 1;
          const int vv = __shfl_sync(0xffffffffu, v, src), dg = __shfl_sync(0xffffffffu, deg, src);
          const int dd = __shfl_sync(0xffffffffu, d, src);
          const int64_t bb = __shfl_sync(0xffffffffu, b, src);
          const long long kk = __shfl_sync(0xffffffffu, Ki, src);
          if (dg > 128 && !SG::kDense) {   // for the block, after the class's other vertices
            if (lane == 0) s_long[atomicAdd(&s_nlong, 1)] = (uint16_t)vv;
            continue;
          }
          int cl[4], cc[4];
          unsigned ww[4];
          auto load = [&](int x0) {   // entries x0 + 32 u + lane of the row
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int x = x0 + u * kWarp + lane;
              cl[u] = vv;
              ww[u] = 0;
              if (x < dg) {
                cl[u] = (int)(__ldg(a.col + bb + x) - v0);
                ww[u] = (unsigned)__ldg(a.wt + bb + x);
              }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) cc[u] = cl[u] != vv ? (int)s.memb[cl[u]] : kEmpty;
          };
          unsigned kid = 0;
          SmallBest best{Arith<false>::lowest(), -1};
          auto candidate = [&](int c, unsigned sum) {
            if (c == dd) {
              kid = sum;
            } else {
              ++cands;
              const long long sc = Arith<false>::score(M, (long long)sum, kk, s.sig[c]);
              if (better(sc, c, best.g, best.c)) best = SmallBest{sc, c};
            }
          };
          load(0);
          if constexpr (SG::kDense) {
            for (int x0 = 0;;) {
#pragma unroll
              for (int u = 0; u < 4; ++u)
                if (cc[u] != kEmpty) atomicAdd(vals + cc[u], ww[u]);
              if ((x0 += 4 * kWarp) >= dg) break;
              load(x0);
            }
            __syncwarp();
            if (dg <= 4 * kWarp) {   // the first lane to take a sum evaluates it
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                const unsigned sum = cc[u] != kEmpty ? atomicExch(vals + cc[u], 0u) : 0u;
                if (sum) candidate(cc[u], sum);
              }
            } else {   // a long row: every community of the graph
              for (int c = lane; c < n; c += kWarp) {
                const unsigned sum = vals[c];
                if (!sum) continue;
                vals[c] = 0;
                candidate(c, sum);
              }
            }
          } else {
            int hs[4];
            const int nu = (dg + kWarp - 1) / kWarp;
            const unsigned fresh = table_add_row<SG::CAP, 4, unsigned>(keys, vals, cc, ww, nu, hs, &ok);
            __syncwarp();
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              if (!((fresh >> u) & 1u)) continue;
              candidate(cc[u], vals[hs[u]]);
              keys[hs[u]] = kEmpty;
              vals[hs[u]] = 0;
            }
          }
          warp_argmax(best.g, best.c);
          kid = __reduce_max_sync(0xffffffffu, kid);
          long long gn = 0;
          if (lane == 0) {
            gn = s.gain(best, dd, kk, M, kid, a.guard);
            if (gn) {
              s.to[vv] = (uint16_t)best.c;
              ++moves;
              S += (u128)(unsigned long long)gn;
            }
          }
          if (a.prune && __shfl_sync(0xffffffffu, gn != 0, 0)) {
            if (lane == 0) s.mark(next, vv);
            if (dg > 4 * kWarp) {
              for (int x = lane; x < dg; x += kWarp) s.mark(next, (int)(__ldg(a.col + bb + x) - v0));
            } else {
#pragma unroll
              for (int u = 0; u < 4; ++u)
                if (cl[u] != vv) s.mark(next, cl[u]);
            }
          }
          __syncwarp();
        }
      }
      __syncthreads();
      // The vertices of degree above 128, queued above, the block together on each.
      // (Finding them by walking the class again cost all 32 warps a list entry
      // and two offsets a vertex: 3,300 pairs beside one vertex of degree 200,
      // one class, 1.07 ms an iteration; with the queue 0.02.)
      const int nlong = s_nlong;
      if (nlong) {   // uniform
        unsigned* dense = s.vals;
        for (int j = 0; j < nlong; ++j) {
          const int v = s_long[j];
          const int64_t b = off[v];
          const int deg = (int)(off[v + 1] - b);
          const int d = s.memb[v];
          const long long Ki = a.K[v0 + v];
          if (tid == 0) s_kid = 0;
          for (int x = tid; x < deg; x += THREADS) {
            const int u = (int)(__ldg(a.col + b + x) - v0);
            if (u != v) atomicAdd(dense + s.memb[u], (unsigned)__ldg(a.wt + b + x));
          }
          __syncthreads();
          SmallBest best{Arith<false>::lowest(), -1};
          for (int x = tid; x < deg; x += THREADS) {   // the first thread to take a sum evaluates it
            const int u = (int)(__ldg(a.col + b + x) - v0);
            if (u == v) continue;
            const int c = s.memb[u];
            const unsigned sum = dense[c] ? atomicExch(dense + c, 0u) : 0u;
            if (!sum) continue;
            if (c == d) {
              s_kid = sum;
            } else {
              ++cands;
              const long long sc = Arith<false>::score(M, (long long)sum, Ki, s.sig[c]);
              if (better(sc, c, best.g, best.c)) best = SmallBest{sc, c};
            }
          }
          warp_argmax(best.g, best.c);
          if (lane == 0) { r_g[wid] = best.g; r_c[wid] = best.c; }
          __syncthreads();
          if (wid == 0) {
            best = lane < NW ? SmallBest{r_g[lane], r_c[lane]} : SmallBest{Arith<false>::lowest(), -1};
            warp_argmax(best.g, best.c);
            if (lane == 0) {
              const long long gn = s.gain(best, d, Ki, M, s_kid, a.guard);
              s_moved = gn != 0;
              if (gn) {
                s.to[v] = (uint16_t)best.c;
                ++moves;
                S += (u128)(unsigned long long)gn;
              }
            }
          }
          __syncthreads();
          if (a.prune && s_moved) {
            if (tid == 0) s.mark(next, v);
            for (int x = tid; x < deg; x += THREADS) s.mark(next, (int)(__ldg(a.col + b + x) - v0));
          }
        }
        __syncthreads();
        if (tid == 0) s_nlong = 0;   // for the next class, after the barrier that ends this one
      }
      // the class's moves
      for (int j = tid; j < m; j += THREADS) {
        const int v = s.list[l0 + j];
        const uint16_t c = s.to[v];
        if (c == SG::kNone) continue;
        s.to[v] = SG::kNone;
        const int d = s.memb[v];
        const long long Ki = a.K[v0 + v];
        s.memb[v] = c;
        shared_add((unsigned long long*)(s.sig + d), (unsigned long long)(-Ki));
        shared_add((unsigned long long*)(s.sig + c), (unsigned long long)Ki);
        atomicSub(s.size + d, 1);
        atomicAdd(s.size + c, 1);
      }
      __syncthreads();
    }
    // the iteration's totals and its stop test
    S = warp_sum_u128(S);
    const unsigned wm = __reduce_add_sync(0xffffffffu, moves);
    if (lane == 0) {
      r_lo[wid] = (unsigned long long)S;
      r_hi[wid] = (unsigned long long)(S >> 64);
      r_moves[wid] = wm;
    }
    __syncthreads();
    if (tid == 0) {
      u128 tot = 0;
      unsigned long long mv = 0;
      for (int w = 0; w < NW; ++w) {
        tot += ((u128)r_hi[w] << 64) | (u128)r_lo[w];
        mv += r_moves[w];
      }
      rec(4 + 3 * it) = mv;
      rec(5 + 3 * it) = (unsigned long long)tot;
      rec(6 + 3 * it) = (unsigned long long)(tot >> 64);
      s_stop = (2.0 * u128_to_double(tot)) / MM <= sa.tol;
    }
    __syncthreads();
    if (s_stop) {
      ++it;
      break;
    }
  }
  for (int v = tid; v < n; v += THREADS) {
    a.memb[v0 + v] = (int32_t)(v0 + s.memb[v]);
    a.sig[v0 + v] = s.sig[v];
    a.csize[v0 + v] = s.size[v];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) edges += __shfl_xor_sync(0xffffffffu, edges, o);
  visited = __reduce_add_sync(0xffffffffu, visited);
  unsigned long long cd = cands;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) cd += __shfl_xor_sync(0xffffffffu, cd, o);
  const bool failed = __syncthreads_or(!ok);
  if (lane == 0) {
    r_lo[wid] = edges;
    r_hi[wid] = visited;
    r_moves[wid] = cd;
  }
  __syncthreads();
  if (tid == 0) {
    unsigned long long e = 0, vs = 0, c = 0;
    for (int w = 0; w < NW; ++w) {
      e += r_lo[w];
      vs += r_hi[w];
      c += r_moves[w];
    }
    rec(0) = failed ? kSmallErr : (unsigned long long)it;
    rec(1) = e;
    rec(2) = vs;
    rec(3) = c;
  }
}

// ----------------------------------------- buckets 3-5: block per vertex

// A decided move waiting for the block to commit it, with its row bounds
// (for the pruning marks).
struct PendingMove {
  int32_t i, c, d, pad;
  int64_t b, e;
};

// Commit and mark the pending moves of a block (all threads take part).
template <typename W, bool ASYNC, bool PULL>
__device__ __forceinline__ void flush_moves(const LMArgs<W>& a, const IterView& iv, const PendingMove* q, int n,
                                            int tid, int nthr) {
  for (int t = tid; t < n; t += nthr) {
    const PendingMove m = q[t];
    if (ASYNC) {
      const long long Ki = a.K[m.i];
      a.memb[m.i] = m.c;
      atomicAdd((unsigned long long*)(a.sig + m.d), (unsigned long long)(-Ki));
      atomicAdd((unsigned long long*)(a.sig + m.c), (unsigned long long)Ki);
      atomicSub(a.csize + m.d, 1);
      atomicAdd(a.csize + m.c, 1);
    } else {
      unsigned long long pos = atomicAdd(a.ctr->nmoves_list + a.odd, 1ull);
      a.moves[pos] = make_int2(m.i, m.c);
    }
  }
  if (!a.prune || (PULL && a.pull_mark)) return;
  if (nthr >= 512) {   // long rows: the whole block marks one after the other
    for (int t = 0; t < n; ++t) mark_row<8>(a, iv, q[t].i, q[t].b, q[t].e, tid, nthr);
  } else {             // one warp per move, the warps' moves in parallel
    for (int t = tid >> 5; t < n; t += nthr >> 5) mark_row<8>(a, iv, q[t].i, q[t].b, q[t].e, tid & 31, kWarp);
  }
}

// Decide (no commit yet): the exact gain of the best candidate against the
// vertex's own community, the guard, and the S / move counts.
// sd, szd: Sigma_d and the size of d, read when the vertex's row was
// (constant within a synchronous class; an asynchronous decision may use any
// recent value).
template <typename W, bool WIDE, bool ASYNC>
__device__ __forceinline__ bool decide_move(const LMArgs<W>& a, BlockAcc& acc, int32_t d, long long Ki, long long sd,
                                            int32_t szd, typename Arith<WIDE>::S best, int32_t c,
                                            unsigned long long kid, long long M, int graph) {
  if (c < 0) return false;
  typedef typename Arith<WIDE>::S S;
  const S g = best - Arith<WIDE>::score(M, (long long)kid, Ki, sd - Ki);
  if (!(g > 0)) return false;
  if (a.guard && c > d && szd == 1 && ld_size<ASYNC>(a.csize + c) == 1) return false;
  const u128 gv = Arith<WIDE>::to_u128(g);
  if (a.gid) {
    atomicAdd(a.g_moves + graph, 1ull);
    atomic_add_u128(a.g_s + 2 * graph, a.g_s + 2 * graph + 1, gv);
  } else {
    atomicAdd(&acc.moves, 1ull);
    atomic_add_u128(&acc.s_lo, &acc.s_hi, gv);
  }
  return true;
}

// One vertex at a time by a block of THREADS threads holding U entries each
// (U * THREADS covers the bucket's largest degree).  As in warp_vertex the
// thread whose entry claims a table slot evaluates and clears it from its own
// registers, so no list of touched slots and no scan of the table is needed.
// Two barriers per vertex: the small shared values alternate between two
// copies by vertex parity, so the next vertex can start while warp 0 still
// decides; moves queue in shared memory and are committed by the whole block
// when the queue fills and at the end.
// Bound by the latency of row, community and total loads and by issue slots
// (R-MAT of 2M vertices, degrees 129-1024: 340 thread instructions an entry
// with the touched-slot list and its scan, 48% of the issue slots).  R-MAT of
// 4.2M vertices, synchronous: 143.4 -> 117.8 ms a run with this kernel, its
// 12288-degree instance in place of the hub chain and 4096-entry hub chunks.
template <typename W, bool WIDE, bool ASYNC, bool PULL, int CAP, int THREADS, int U>
__global__ void __launch_bounds__(THREADS, THREADS <= 128 ? 8 : THREADS <= 512 ? 2 : 1)
    lm_block(LMArgs<W> a, const int32_t* __restrict__ list, const int64_t* __restrict__ ko) {
  const IterView iv = iter_view(a);
  if (iv.iter < 0) return;
  const int32_t* __restrict__ verts = list + ko[0];
  const int nverts = (int)(ko[1] - ko[0]);
  typedef typename Arith<WIDE>::S S;
  typedef typename TableVal<WIDE>::T V;
  constexpr int NW = THREADS / kWarp;
  constexpr int LD = ASYNC ? 1 : 0;
  constexpr int QCAP = 64;
  // dynamic shared memory: values (CAP V), keys (CAP i32)
  extern __shared__ unsigned long long dyn[];
  V* vals = (V*)dyn;
  int32_t* keys = (int32_t*)(vals + CAP);
  __shared__ BlockAcc acc;
  __shared__ S red_g[2][NW];
  __shared__ int32_t red_c[2][NW];
  __shared__ unsigned long long s_kid[2];
  __shared__ PendingMove queue[QCAP];
  __shared__ int q_n;
  __shared__ VertexRow win[kWarp];
  __shared__ unsigned s_live[2];   // by window parity: an empty window has no other barrier
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  acc_init(acc);
  if (threadIdx.x == 0) { s_kid[0] = s_kid[1] = 0; q_n = 0; }
  for (int t = threadIdx.x; t < CAP; t += THREADS) { keys[t] = kEmpty; vals[t] = 0; }
  __syncthreads();
  bool ok = true;
  int p = 0, wp = 0;
  WarpTally tally;
  // the next 32 vertices, loaded by warp 0 (in shared memory: a row's bounds,
  // community and degree are read where they are used instead of held)
  for (int64_t w0 = blockIdx.x; w0 < nverts; w0 += (int64_t)kWarp * gridDim.x, wp ^= 1) {
    if (wid == 0) {
      VertexRow r;
      const unsigned on = vertex_window<W, PULL>(a, iv, verts, nverts, w0, gridDim.x, lane, r);
      if (!(PULL && a.pull_check) && ((on >> lane) & 1u)) {
        tally.edges += (unsigned)r.deg;
        ++tally.visited;
      }
      win[lane] = r;
      if (lane == 0) s_live[wp] = on;
    }
    __syncthreads();
    for (unsigned live = s_live[wp]; live; live &= live - 1) {   // uniform across the block
      const VertexRow& v = win[__ffs(live) - 1];
      long long sd = 0;
      int32_t szd = 0;
      if (wid == 0) {   // for the decision
        sd = ld_state<LD>(a.sig + word_id<PULL>(v.d));
        szd = ld_state<LD>(a.csize + word_id<PULL>(v.d));
      }
      // this warp's rounds that hold at least one entry (the rest skipped)
      const int rem = v.deg - wid * kWarp;
      const int nu = rem <= 0 ? 0 : (rem + THREADS - 1) / THREADS;
      int32_t cc[U];
      int hs[U];
      unsigned fresh;
      int32_t seen = 0;
      {
        V ww[U];
        seen = row_communities<U, LD, PULL>(a, v, (int)threadIdx.x, THREADS, nu, cc, ww);
        fresh = table_add_row<CAP, U, V>(keys, vals, cc, ww, nu, hs, &ok);
      }
      // B1: table complete; warp 0 has finished the previous vertex
      if (PULL && a.pull_check) {
        const bool on = __syncthreads_or(((seen | v.d) & moved_bit(iv.iter - 1)) != 0);
        if (!on) {   // not active after all: the table is cleared and nothing else done
#pragma unroll
          for (int u = 0; u < U; ++u)
            if ((fresh >> u) & 1u) {
              keys[hs[u]] = kEmpty;
              vals[hs[u]] = 0;
            }
          __syncthreads();
          continue;
        }
        if (threadIdx.x == 0) {
          tally.edges += (unsigned)v.deg;
          ++tally.visited;
        }
      } else {
        __syncthreads();
      }
      if (q_n >= QCAP) {   // uniform: q_n was last written before this barrier
        flush_moves<W, ASYNC, PULL>(a, iv, queue, q_n, threadIdx.x, THREADS);
        __syncthreads();
        if (threadIdx.x == 0) q_n = 0;
      }
      if (threadIdx.x == 0) s_kid[p ^ 1] = 0;   // the next vertex's copy
      const long long M = a.gid ? a.Mg[a.gid[v.i]] : a.M, Ki = v.Ki;
      const int32_t d = word_id<PULL>(v.d);
      S bg = Arith<WIDE>::lowest();
      int32_t bc = -1;
#pragma unroll
      for (int u0 = 0; u0 < U; u0 += 4) {
        if (u0 >= nu) break;
        long long sg[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
          sg[j] = ((fresh >> (u0 + j)) & 1u) && cc[u0 + j] != d ? ld_state<LD>(a.sig + cc[u0 + j]) : 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int u = u0 + j;
          if (!((fresh >> u) & 1u)) continue;
          const V sum = vals[hs[u]];
          if (cc[u] != d) {
            ++tally.cands;
            const S g = Arith<WIDE>::score(M, (long long)sum, Ki, sg[j]);
            if (better(g, cc[u], bg, bc)) { bg = g; bc = cc[u]; }
          } else {
            s_kid[p] = sum;
          }
          keys[hs[u]] = kEmpty;
          vals[hs[u]] = 0;
        }
      }
      warp_argmax(bg, bc);
      if (lane == 0) { red_g[p][wid] = bg; red_c[p][wid] = bc; }
      __syncthreads();   // B2: candidates evaluated, table clear
      if (wid == 0) {
        bg = lane < NW ? red_g[p][lane] : Arith<WIDE>::lowest();
        bc = lane < NW ? red_c[p][lane] : -1;
        warp_argmax(bg, bc);
        if (lane == 0 &&
            decide_move<W, WIDE, ASYNC>(a, acc, d, Ki, sd, szd, bg, bc, s_kid[p], M, a.gid ? a.gid[v.i] : 0))
          queue[q_n++] = PendingMove{v.i, bc, d, 0, v.b, v.b + v.deg};
      }
      p ^= 1;
    }
  }
  tally.add(acc);
  __syncthreads();
  flush_moves<W, ASYNC, PULL>(a, iv, queue, q_n, threadIdx.x, THREADS);
  if (!ok) atomicOr(&acc.error, kErrProbe);
  __syncthreads();
  acc_flush(acc, a.ctr);
}

// ------------------------------------------------- bucket 6: hub vertices
//
// Hub h of a class owns global table slots [hbase[h] - hbase[0], + 2 deg):
// every class's tables start at slot 0, so a class reuses the slots the
// previous class's scan just cleared, which are still in L2.
// 1. insert: blocks are (hub, a.hchunk-entry chunk) pairs; each sums its chunk
//    per community in shared memory, then adds each distinct community once
//    to the hub's global table;
// 2. scan: blocks are (hub, 4096-slot chunk) pairs; each evaluates the gain
//    of every occupied slot, clears it, and leaves its chunk's best (and
//    K_{i->d} of the slot holding d); the last block of a hub reduces the
//    chunk bests and commits;
// 3. mark (once per iteration, all classes): neighbours of the hubs that moved.

constexpr int kItemCache = 512;   // hub prefix entries a block copies to shared memory

template <typename W, bool WIDE, bool ASYNC, bool PULL, int CHUNK, int THREADS>
__global__ void __launch_bounds__(THREADS) lm_hub_insert(LMArgs<W> a, const int32_t* __restrict__ hubs, int nhubs,
                                                         const int64_t* __restrict__ chunk_pre) {
  typedef typename TableVal<WIDE>::T V;
  const IterView iv = iter_view(a);
  if (iv.iter < 0) return;
  constexpr int CAP = 2 * CHUNK;
  constexpr int U = CHUNK / THREADS;
  static_assert(U >= 1 && CHUNK % THREADS == 0, "a chunk covers whole rounds of the block");
  extern __shared__ unsigned long long hdyn[];
  V* svals = (V*)hdyn;
  int32_t* skeys = (int32_t*)(svals + CAP);
  __shared__ int64_t s_pre[kItemCache + 1];
  const int h = block_item<kItemCache>(chunk_pre, nhubs, blockIdx.x, s_pre);
  VertexRow v;
  v.i = hubs[h];
  if (!is_active<PULL>(a, iv, v.i)) return;   // uniform across the block
  if (!graph_of(a, v.i, &v.M, &v.graph)) return;
  const int64_t q = (int64_t)blockIdx.x - (chunk_pre[h] - chunk_pre[0]);
  for (int t = threadIdx.x; t < CAP; t += THREADS) { skeys[t] = kEmpty; svals[t] = 0; }
  __syncthreads();
  const int64_t b = a.off[v.i], e = a.off[v.i + 1];
  const int64_t base = a.hbase[h] - a.hbase[0];   // the class's tables start at slot 0
  const uint32_t cap = (uint32_t)(2 * (e - b));
  v.b = b + q * CHUNK;
  v.deg = (int)min((int64_t)CHUNK, e - v.b);
  bool ok = true;
  int32_t cc[U];
  V ww[U];
  int hs[U];
  const int32_t seen = row_communities<U, (ASYNC ? 1 : 0), PULL>(a, v, (int)threadIdx.x, THREADS, U, cc, ww);
  // a neighbour moved: the scan finds the hub active
  if (PULL && a.pull_check && __any_sync(0xffffffffu, (seen & moved_bit(iv.iter - 1)) != 0) && (threadIdx.x & 31) == 0)
    a.hmoved[h] = -(iv.iter + 1);
  const unsigned fresh = table_add_row<CAP, U, V>(skeys, svals, cc, ww, U, hs, &ok);
  __syncthreads();
  // the thread that claimed a slot adds its sum to the hub's table
  unsigned long long vv[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const bool mine = (fresh >> u) & 1u;
    vv[u] = mine ? (unsigned long long)svals[hs[u]] : 0ull;
    if (!mine) cc[u] = kEmpty;
  }
  ok &= gtable_add_many<U>(a.hkeys + base, a.hvals + base, cap, cc, vv);
  if (!ok) atomicOr(&a.ctr->error, kErrProbe);
}

// Scan blocks are (hub, kSlotChunk-slot chunk) pairs: each evaluates the
// gain of every occupied slot of its chunk, clears it, and leaves its chunk's
// best; the block that finishes a hub's last chunk (a per-hub counter after a
// fence) reduces the hub's chunk bests and commits the hub's move, so the
// decision needs no launch of its own.  No block waits for another.
template <typename W, bool WIDE, bool ASYNC, bool PULL>
__global__ void __launch_bounds__(256) lm_hub_scan(LMArgs<W> a, const int32_t* __restrict__ hubs, int nhubs) {
  const IterView iv = iter_view(a);
  if (iv.iter < 0) return;
  typedef typename Arith<WIDE>::S S;
  constexpr int NW = 256 / kWarp;
  __shared__ S red_g[NW];
  __shared__ int32_t red_c[NW];
  __shared__ unsigned red_n[NW];
  __shared__ BlockAcc acc;
  __shared__ int s_last;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __shared__ int64_t s_pre[kItemCache + 1];
  const int h = block_item<kItemCache>(a.spre, nhubs, blockIdx.x, s_pre);
  const int32_t i = hubs[h];
  if (!is_active<PULL>(a, iv, i)) return;   // uniform across the block
  long long M;
  int graph;
  if (!graph_of(a, i, &M, &graph)) return;
  acc_init(acc);
  const int64_t q = (int64_t)blockIdx.x - (a.spre[h] - a.spre[0]);
  const int64_t b = a.off[i], e = a.off[i + 1];
  const int64_t cap = 2 * (e - b);
  const int64_t base = a.hbase[h] - a.hbase[0];
  const int32_t dw = a.memb[i], d = word_id<PULL>(dw);
  const bool on = !(PULL && a.pull_check) || (dw & moved_bit(iv.iter - 1)) || a.hmoved[h] == -(iv.iter + 1);
  const long long Ki = a.K[i];
  const int64_t t0 = q * kSlotChunk, t1 = min(cap, t0 + kSlotChunk);
  S bg = Arith<WIDE>::lowest();
  int32_t bc = -1;
  unsigned ncand = 0;
  constexpr int U = 4;
  for (int64_t y = t0; y < t1; y += U * 256) {
    int32_t cs[U];
    unsigned long long vs[U];
    long long sg[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t t = y + u * 256 + threadIdx.x;
      cs[u] = t < t1 ? a.hkeys[base + t] : kEmpty;
      vs[u] = cs[u] != kEmpty ? a.hvals[base + t] : 0ull;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) sg[u] = (cs[u] != kEmpty && cs[u] != d) ? ld_sig<ASYNC>(a.sig + cs[u]) : 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (cs[u] == kEmpty) continue;
      const int64_t t = y + u * 256 + threadIdx.x;
      if (PULL && !on) {   // inactive after all: only cleared
      } else if (cs[u] != d) {
        ++ncand;
        S g = Arith<WIDE>::score(M, (long long)vs[u], Ki, sg[u]);
        if (better(g, cs[u], bg, bc)) { bg = g; bc = cs[u]; }
      } else {
        a.hkid[h] = vs[u];   // K_{i->d}; only one slot holds d
      }
      a.hkeys[base + t] = kEmpty;
      a.hvals[base + t] = 0;
    }
  }
  ncand = __reduce_add_sync(0xffffffffu, ncand);
  warp_argmax(bg, bc);
  if (lane == 0) { red_g[wid] = bg; red_c[wid] = bc; red_n[wid] = ncand; }
  __syncthreads();
  if (wid == 0) {
    bg = lane < NW ? red_g[lane] : Arith<WIDE>::lowest();
    bc = lane < NW ? red_c[lane] : -1;
    warp_argmax(bg, bc);
    ncand = __reduce_add_sync(0xffffffffu, lane < NW ? red_n[lane] : 0u);
    if (lane == 0) {
      if (ncand) atomicAdd(&a.ctr->cands, (unsigned long long)ncand);
      const int64_t slot = a.spre[h] + q;
      u128 gu = (u128)(i128)bg;
      a.hpart[2 * slot] = (long long)(unsigned long long)gu;
      a.hpart[2 * slot + 1] = (long long)(unsigned long long)(gu >> 64);
      a.hpart_c[slot] = bc;
      __threadfence();   // the chunk best (and K_{i->d}) before the count
      const int nck = (int)(a.spre[h + 1] - a.spre[h]);
      s_last = atomicAdd(a.hdone + h, 1) == nck - 1;
    }
  }
  __syncthreads();
  if (s_last && wid == 0) {   // every chunk of this hub is done: decide
    __threadfence();
    S hg = Arith<WIDE>::lowest();
    int32_t hc = -1;
    for (int64_t t = a.spre[h] + lane; t < a.spre[h + 1]; t += kWarp) {
      const i128 g = ((i128)__ldcg(a.hpart + 2 * t + 1) << 64) | (i128)(unsigned long long)__ldcg(a.hpart + 2 * t);
      const int32_t c = __ldcg(a.hpart_c + t);
      if (c >= 0 && better((S)g, c, hg, hc)) { hg = (S)g; hc = c; }
    }
    warp_argmax(hg, hc);
    if (lane == 0) {
      if (on) {
        atomicAdd(&acc.edges, (unsigned long long)(e - b));
        atomicAdd(&acc.visited, 1ull);
      }
      const bool moved = on && commit_choice<W, WIDE, ASYNC>(a, acc, i, d, Ki, ld_sig<ASYNC>(a.sig + d),
                                                       ld_size<ASYNC>(a.csize + d), hg, hc, __ldcg(a.hkid + h), M,
                                                       graph);
      a.hkid[h] = 0;
      a.hdone[h] = 0;
      if (moved && a.prune && !(PULL && a.pull_mark)) a.hmoved[h] = iv.iter + 1;   // lm_hub_mark marks its neighbours
    }
  }
  __syncthreads();
  acc_flush(acc, a.ctr);
}

// Pruning marks of the hubs that moved in this iteration (all classes at
// once; the marks only feed the next iteration's active set): blocks are
// (hub, a.hchunk-entry chunk) pairs of the pass's whole hub list.
template <typename W>
__global__ void __launch_bounds__(256) lm_hub_mark(LMArgs<W> a, const int32_t* __restrict__ hubs, int nhubs,
                                                   const int64_t* __restrict__ chunk_pre) {
  const IterView iv = iter_view(a);
  if (iv.iter < 0) return;
  __shared__ int64_t s_pre[kItemCache + 1];
  const int h = block_item<kItemCache>(chunk_pre, nhubs, blockIdx.x, s_pre);
  if (a.hmoved[h] != iv.iter + 1) return;
  const int32_t i = hubs[h];
  const int64_t q = (int64_t)blockIdx.x - (chunk_pre[h] - chunk_pre[0]);
  const int64_t b = a.off[i], e = a.off[i + 1];
  const int64_t x0 = b + q * a.hchunk, x1 = min(e, x0 + a.hchunk);
  if (q == 0 && threadIdx.x == 0) iv.sw[i] = iv.iter + 1;
  mark_row<4>(a, iv, i, x0, x1, (int)threadIdx.x, 256, false);   // the hub itself: marked above
}

// ----------------------------------------------- synchronous commit step

// It also clears the next class's counter (free: the class before this one,
// which used it last, is committed).
template <typename W>
__global__ void __launch_bounds__(256) lm_commit(LMArgs<W> a) {
  const unsigned long long n = a.ctr->nmoves_list[a.odd];
  const bool pull = a.pull_check || a.pull_mark;
  // the flag of this iteration's moves, and the last one's, which later classes read
  const int it = *a.d_iter;
  const int32_t flag = a.pull_mark ? moved_bit(it) : 0, kept = a.pull_check ? moved_bit(it - 1) : 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) a.ctr->nmoves_list[a.odd ^ 1] = 0;
  for (unsigned long long t = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; t < n;
       t += (unsigned long long)gridDim.x * blockDim.x) {
    int2 mv = a.moves[t];
    // both loads before the store (a load after it would wait for the first):
    // road grid of 16.8M vertices 34.3 -> 30.2 ms a run
    const int32_t i = mv.x, c = mv.y, w = a.memb[i], d = pull ? w & kIdMask : w;
    const long long Ki = a.K[i];
    a.memb[i] = c | flag | (w & kept);
    atomicAdd((unsigned long long*)(a.sig + d), (unsigned long long)(-Ki));
    atomicAdd((unsigned long long*)(a.sig + c), (unsigned long long)Ki);
    atomicSub(a.csize + d, 1);
    atomicAdd(a.csize + c, 1);
  }
}

// memb &= keep (flags that have been read; both at the end of a phase).
__global__ void clear_flags_k(int32_t* __restrict__ memb, int64_t n, int32_t keep) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t w = memb[i];
    if ((w & keep) != w) memb[i] = w & keep;
  }
}
void lm_clear_flags(int32_t* memb, int64_t n, int iter, cudaStream_t s) {
  const int32_t keep = iter < 0 ? kIdMask : (iter & 1) ? 0x7fffffff : (int32_t)0xbfffffff;
  const unsigned blocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 16));
  (count_launch(), clear_flags_k<<<blocks, 256, 0, s>>>(memb, n, keep));
}

// The end of an iteration of one graph, on the device: its counters go to
// slot (iteration mod 4) of hist (pinned host memory: no copy to queue) and are
// cleared for the next one, and the iteration number moves on, or to -1
// when the phase ends (the stop test of the host, on the same roundings), which
// makes the launches of an iteration queued behind it return at once.
__global__ void lm_decide_k(DevCounters* ctr, DevCounters* hist, int* d_iter, double MM, double tol) {
  const int it = *d_iter;
  if (it < 0) return;
  hist[it & 3] = *ctr;
  const u128 S = ((u128)ctr->s_hi << 64) | (u128)ctr->s_lo;
  *d_iter = (2.0 * u128_to_double(S)) / MM <= tol ? -1 : it + 1;
  memset(ctr, 0, sizeof(DevCounters));
}
void lm_decide(DevCounters* ctr, DevCounters* hist, int* d_iter, double MM, double tol, cudaStream_t s) {
  (count_launch(), lm_decide_k<<<1, 1, 0, s>>>(ctr, hist, d_iter, MM, tol));
}

// ---------------------------------------------------------------- launch

namespace {

template <typename K>
int grid_for(K kernel, int threads, size_t smem, int64_t work_blocks) {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 1;
  }
  const int per_sm = blocks_per_sm(kernel, threads, smem);
  int g = sms * per_sm;
  if (work_blocks < g) g = (int)work_blocks;
  return g < 1 ? 1 : g;
}

template <typename W, bool WIDE, bool ASYNC, bool PULL, int CAP, int THREADS, int U>
void launch_block_t(const LMArgs<W>& a, const int32_t* list, const int64_t* ko, int64_t nverts, cudaStream_t s) {
  const size_t smem = (size_t)CAP * (sizeof(typename TableVal<WIDE>::T) + 4);
  auto k = lm_block<W, WIDE, ASYNC, PULL, CAP, THREADS, U>;
  static std::atomic<unsigned long long> attr{0};
  smem_limit_once(attr, k, smem);
  (count_launch(), k<<<grid_for(k, THREADS, smem, nverts), THREADS, smem, s>>>(a, list, ko));
}

template <typename W, bool WIDE, bool ASYNC, bool PULL>
void launch_bucket_t(const LMArgs<W>& a, int bucket, const int32_t* list, const int64_t* ko, int64_t nverts, cudaStream_t s) {
  if (nverts <= 0) return;
  switch (bucket) {
    case 0: {
      auto k = lm_thread<W, WIDE, ASYNC, PULL>;
      (count_launch(), k<<<grid_for(k, 256, 0, (nverts + 255) / 256), 256, 0, s>>>(a, list, ko));
      break;
    }
    case 1: {
      if constexpr (!WIDE) {   // narrow sums: a lane per vertex, its row sorted in registers
        auto k = lm_thread_sorted<W, ASYNC, PULL, 32>;
        (count_launch(), k<<<grid_for(k, 128, 0, (nverts + 127) / 128), 128, 0, s>>>(a, list, ko));
      } else {
        auto k = lm_warp<W, WIDE, ASYNC, PULL, 64, 1>;
        (count_launch(), k<<<grid_for(k, 256, 0, (nverts + 7) / 8), 256, 0, s>>>(a, list, ko));
      }
      break;
    }
    case 2: {
      auto k = lm_warp<W, WIDE, ASYNC, PULL, 256, 4>;
      (count_launch(), k<<<grid_for(k, 256, 0, (nverts + 7) / 8), 256, 0, s>>>(a, list, ko));
      break;
    }
    case 3: launch_block_t<W, WIDE, ASYNC, PULL, 2048, 128, 8>(a, list, ko, nverts, s); break;
    case 4: launch_block_t<W, WIDE, ASYNC, PULL, 8192, 512, 8>(a, list, ko, nverts, s); break;
    case 5: launch_block_t<W, WIDE, ASYNC, PULL, 18432, 1024, 12>(a, list, ko, nverts, s); break;
    default: break;
  }
}

}  // namespace

template <typename W>
void lm_launch_bucket(const LMArgs<W>& a, bool wide, bool async, int bucket, const int32_t* list, const int64_t* ko,
                      int64_t nverts, cudaStream_t s) {
  const bool pull = a.pull_check || a.pull_mark;   // synchronous only
  if (wide) {
    if (async) launch_bucket_t<W, true, true, false>(a, bucket, list, ko, nverts, s);
    else if (pull) launch_bucket_t<W, true, false, true>(a, bucket, list, ko, nverts, s);
    else launch_bucket_t<W, true, false, false>(a, bucket, list, ko, nverts, s);
  } else {
    if (async) launch_bucket_t<W, false, true, false>(a, bucket, list, ko, nverts, s);
    else if (pull) launch_bucket_t<W, false, false, true>(a, bucket, list, ko, nverts, s);
    else launch_bucket_t<W, false, false, false>(a, bucket, list, ko, nverts, s);
  }
}

template <typename W, bool WIDE, bool ASYNC, bool PULL, int CHUNK, int THREADS>
static void launch_hub_insert_t(const LMArgs<W>& a, const int32_t* hubs, int nhubs, const int64_t* chunk_pre,
                                int64_t nchunks, cudaStream_t s) {
  const size_t smem = (size_t)(2 * CHUNK) * (sizeof(typename TableVal<WIDE>::T) + 4);
  auto k = lm_hub_insert<W, WIDE, ASYNC, PULL, CHUNK, THREADS>;
  static std::atomic<unsigned long long> attr{0};
  smem_limit_once(attr, k, smem);
  (count_launch(), k<<<(unsigned)nchunks, THREADS, smem, s>>>(a, hubs, nhubs, chunk_pre));
}

template <typename W, bool WIDE, bool ASYNC, bool PULL>
static void launch_hubs_t(const LMArgs<W>& a, const int32_t* hubs, int nhubs, const int64_t* chunk_pre,
                          int64_t nchunks, int64_t nslotchunks, cudaStream_t s) {
  if (a.hchunk == kHubLongChunk)
    launch_hub_insert_t<W, WIDE, ASYNC, PULL, kHubLongChunk, 512>(a, hubs, nhubs, chunk_pre, nchunks, s);
  else
    launch_hub_insert_t<W, WIDE, ASYNC, PULL, kHubShortChunk, 256>(a, hubs, nhubs, chunk_pre, nchunks, s);
  (count_launch(), lm_hub_scan<W, WIDE, ASYNC, PULL><<<(unsigned)nslotchunks, 256, 0, s>>>(a, hubs, nhubs));
}

template <typename W>
void lm_launch_hubs(const LMArgs<W>& a, bool wide, bool async, const int32_t* hubs, int nhubs,
                    const int64_t* chunk_pre, int64_t nchunks, const int64_t* spre, int64_t nslotchunks,
                    cudaStream_t s) {
  if (nhubs <= 0 || nchunks <= 0) return;
  const bool pull = a.pull_check || a.pull_mark;   // synchronous only
  if (wide) {
    if (async) launch_hubs_t<W, true, true, false>(a, hubs, nhubs, chunk_pre, nchunks, nslotchunks, s);
    else if (pull) launch_hubs_t<W, true, false, true>(a, hubs, nhubs, chunk_pre, nchunks, nslotchunks, s);
    else launch_hubs_t<W, true, false, false>(a, hubs, nhubs, chunk_pre, nchunks, nslotchunks, s);
  } else {
    if (async) launch_hubs_t<W, false, true, false>(a, hubs, nhubs, chunk_pre, nchunks, nslotchunks, s);
    else if (pull) launch_hubs_t<W, false, false, true>(a, hubs, nhubs, chunk_pre, nchunks, nslotchunks, s);
    else launch_hubs_t<W, false, false, false>(a, hubs, nhubs, chunk_pre, nchunks, nslotchunks, s);
  }
}

template <typename W>
void lm_launch_class(const LMArgs<W>& a, bool wide, bool async, const int32_t* list, const int64_t* ko, int P,
                     int ch, int64_t nverts, cudaStream_t s) {
  if (nverts <= 0) return;
  int64_t blocks = (nverts + 7) / 8;
  if (blocks > 152 * 3) blocks = 152 * 3;   // resident blocks (three per SM)
  const unsigned g = (unsigned)blocks;
  if (wide) {
    if (async) (count_launch(), lm_class<W, true, true><<<g, 256, 0, s>>>(a, list, ko, P, ch));
    else (count_launch(), lm_class<W, true, false><<<g, 256, 0, s>>>(a, list, ko, P, ch));
  } else {
    if (async) (count_launch(), lm_class<W, false, true><<<g, 256, 0, s>>>(a, list, ko, P, ch));
    else (count_launch(), lm_class<W, false, false><<<g, 256, 0, s>>>(a, list, ko, P, ch));
  }
}

namespace {

template <typename W, int NMAX, int THREADS>
void launch_small_t(const LMArgs<W>& a, const SmallArgs& sa, cudaStream_t s) {
  auto k = lm_small<W, NMAX, THREADS>;
  const size_t smem = SmallGraph<W, NMAX, THREADS>::kBytes;
  static std::atomic<unsigned long long> attr{0};
  smem_limit_once(attr, k, smem);
  (count_launch(), k<<<(unsigned)sa.count, THREADS, smem, s>>>(a, sa));
}

}  // namespace

// Graphs of at most kTinyVerts vertices take 256 threads and 51 KB (four
// blocks on an SM), larger ones a whole SM.
template <typename W>
void lm_launch_small(const LMArgs<W>& a, const SmallArgs& sa, cudaStream_t s) {
  if (sa.count <= 0) return;
  if (sa.tiny) launch_small_t<W, kTinyVerts, 256>(a, sa, s);
  else launch_small_t<W, kSmallVerts, 1024>(a, sa, s);
}

template <typename W>
void lm_launch_hub_mark(const LMArgs<W>& a, const int32_t* hubs, int nhubs, const int64_t* chunk_pre, int64_t nchunks,
                        cudaStream_t s) {
  if (nhubs <= 0 || nchunks <= 0 || !a.prune || a.pull_mark) return;
  (count_launch(), lm_hub_mark<W><<<(unsigned)nchunks, 256, 0, s>>>(a, hubs, nhubs, chunk_pre));
}

template <typename W>
void lm_launch_commit(const LMArgs<W>& a, int64_t max_moves, cudaStream_t s) {
  if (max_moves <= 0) return;
  int blocks = (int)((max_moves + 255) / 256);
  if (blocks > 152 * 16) blocks = 152 * 16;
  (count_launch(), lm_commit<W><<<blocks, 256, 0, s>>>(a));
}

template void lm_launch_bucket<int32_t>(const LMArgs<int32_t>&, bool, bool, int, const int32_t*, const int64_t*,
                                        int64_t, cudaStream_t);
template void lm_launch_bucket<int64_t>(const LMArgs<int64_t>&, bool, bool, int, const int32_t*, const int64_t*,
                                        int64_t, cudaStream_t);
template void lm_launch_hubs<int32_t>(const LMArgs<int32_t>&, bool, bool, const int32_t*, int, const int64_t*,
                                      int64_t, const int64_t*, int64_t, cudaStream_t);
template void lm_launch_hubs<int64_t>(const LMArgs<int64_t>&, bool, bool, const int32_t*, int, const int64_t*,
                                      int64_t, const int64_t*, int64_t, cudaStream_t);
template void lm_launch_class<int32_t>(const LMArgs<int32_t>&, bool, bool, const int32_t*, const int64_t*, int,
                                       int, int64_t, cudaStream_t);
template void lm_launch_class<int64_t>(const LMArgs<int64_t>&, bool, bool, const int32_t*, const int64_t*, int,
                                       int, int64_t, cudaStream_t);
template void lm_launch_small<int32_t>(const LMArgs<int32_t>&, const SmallArgs&, cudaStream_t);
template void lm_launch_small<int64_t>(const LMArgs<int64_t>&, const SmallArgs&, cudaStream_t);
template void lm_launch_hub_mark<int32_t>(const LMArgs<int32_t>&, const int32_t*, int, const int64_t*, int64_t,
                                          cudaStream_t);
template void lm_launch_hub_mark<int64_t>(const LMArgs<int64_t>&, const int32_t*, int, const int64_t*, int64_t,
                                          cudaStream_t);
template void lm_launch_commit<int32_t>(const LMArgs<int32_t>&, int64_t, cudaStream_t);
template void lm_launch_commit<int64_t>(const LMArgs<int64_t>&, int64_t, cudaStream_t);

}  // namespace gbl
