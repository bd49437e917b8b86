// sweep.cu -- colour-class steps of the deterministic local-moving phase in one persistent launch.
//
// The colour-synchronous schedule runs one step per colour class (hundreds on a graph with hubs, a
// handful of vertices each in the late ones): every flagged vertex of the class decides against the
// class-start totals, then all moves apply.  As separate launches such a step costs a fork to the
// degree buckets' streams, their join, the apply kernel and, with giant rows, four more kernels one
// after another: 7 us for a step with almost no work, 47 us for a hub's.  Here the whole phase (or an
// iteration's narrow classes, where a graph also has wide ones) is one launch whose blocks stay
// resident, and what a step costs is one barrier and one chain of dependent loads (list entry, row
// bounds, arcs, C'[j], Sigma_c).  So
//   * a row of every bucket fits its group in one step: 4 lanes to 4 arcs (no table: lanes compare
//     their communities by shuffles), 8 lanes to 16, a warp to 128, 128 threads to 512, 512 to 2048,
//     1024 to 4096, so nothing loops over a row and its targets are still in registers when a move
//     marks its neighbours; the tables of all group sizes are slices of one 8192-slot table;
//   * the lane that claims a slot scores and clears it: its Sigma_c load is issued at the claim;
//   * Sigma is kept twice.  A step reads one copy and adds its moves to the other; the next step
//     swaps them and first repeats those moves (kept in shared memory) on the copy that lacks them.
//     So a step needs no second barrier between deciding and applying.  A step with more vertices
//     than a block can keep decides, waits, and applies to both copies;
//   * giant rows: arcs insert into the shared pool by the warp, a barrier, 128 threads score 1024
//     slots, a barrier, and every warp that marks a giant's arcs reduces the giant's candidates
//     itself; both are skipped when no giant of the class is flagged;
//   * the tolerance test is made by every block from sums that come with the last step's barrier.
// Integer results are those of the separate kernels bit for bit (exact sums, ties by id).
#include <atomic>

#include "giant.cuh"
#include "persist.cuh"

namespace lv {

// Table slots of a block, divided among its groups: four per arc of the longest row of a bucket (half
// full, a 4096-arc row's insertion takes 11,000 cycles of probing against 4,000), two per arc of the
// longest row a block takes.
constexpr int kSwSlots = 16384;
constexpr int kSwLongest = 8192;   // giant rows up to this are a block's, longer ones the whole launch's
constexpr int kSwMoves = kSweepMoves;
constexpr int kSwWarps = kPersistThreads / 32;

template <class M>
struct SweepArgs {
  GraphView<typename M::w_t> g;
  PassState<M> st;
  typename M::a_t* sig2;      // second copy of st.Sig
  int64_t n_sig;              // its entries
  const int32_t* perm;
  const int32_t* glist;       // class-ordered giant list (base of the records' offset)
  const int64_t* recs;        // step records
  int nsteps;
  int whole;                  // 1: every iteration until the phase ends; 0: one iteration's steps
  int pruning;
  int n_graphs;
  int all_wide;               // 1: the launch has fewer blocks than the records were made for
  GiantPlan gp;
  unsigned long long* state;  // kSw* below, zeroed before the launch
};
// 3 barrier words, then 3 rotating sums of an iteration {lo, hi, fp, moves}
enum { kSwBar = 0, kSwSums = 4, kSwWords = kSwSums + 12 };
static_assert(kSwWords <= kSweepStateWords, "state block");

template <class M>
struct SweepMove {
  int32_t from, to;
  typename M::a_t k;
};

template <class M>
struct SweepShared {
  int32_t keys[kSwSlots];
  typename M::h_t vals[kSwSlots];
  SweepMove<M> moves[2][kSwMoves];
  int n_moves[3];
  int64_t rec[2][kStepWords];
  typename M::s_t red_s[kSwWarps];
  int32_t red_c[kSwWarps];
  typename M::h_t red_h[kSwWarps];
  unsigned long long lo, hi, mv;  // this block's sums of the iteration
  double f;
  int done, act;
};

// A group of G threads: lanes of a warp, or whole warps that meet at a named barrier (128-thread groups
// 1-8, 512-thread groups 9-10, the block 0).
template <int G>
__device__ __forceinline__ void team_sync() {
  if constexpr (G < 32) __syncwarp(Grp<G>::mask());
  else if constexpr (G == 32) __syncwarp();
  else if constexpr (G == kPersistThreads) __syncthreads();
  else {
    const int id = (G == 128 ? 1 : 9) + (int)threadIdx.x / G;
    asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(G) : "memory");
  }
}

// Whether any thread of the group says so: the same answer on all of them, whatever changes meanwhile.
template <int G>
__device__ __forceinline__ bool team_any(bool p) {
  if constexpr (G <= 32) return __any_sync(Grp<G>::mask(), p);
  else if constexpr (G == kPersistThreads) return __syncthreads_or(p ? 1 : 0) != 0;
  else {
    const int id = (G == 128 ? 1 : 9) + (int)threadIdx.x / G;
    int r;
    asm volatile("{\n\t.reg .pred q, r;\n\tsetp.ne.s32 q, %1, 0;\n\tbar.red.or.pred r, %2, %3, q;\n\tselp.s32 %0, 1, 0, r;\n\t}"
                 : "=r"(r) : "r"((int)p), "r"(id), "n"(G) : "memory");
    return r != 0;
  }
}

// What the row code costs is instructions (a block of 32 warps shares four issue slots), so it counts
// them: one compare-and-swap a probe instead of a read, a compare and a swap; the value is added
// once, after the probing; arg-max and sums by the warp reduction unit; 32-bit factors in the score.

// Adds (key, w) to a table of mask + 1 slots, at most half full; *own = this call claimed the slot.
// Returns the slot (mask + 1 if the table was full, which its size excludes).
template <class V>
__device__ __forceinline__ unsigned tbl_put(int32_t* keys, V* vals, unsigned mask, int shift, int32_t key, V w, bool* own) {
  unsigned s = tbl_home(key, shift);
  int32_t old = 0;
  unsigned left = mask + 1;
  do {
    old = atomicCAS(&keys[s], kEmpty, key);
    if (old == kEmpty || old == key) break;
    s = (s + 1) & mask;
  } while (--left);
  *own = old == kEmpty;
  if (left == 0) return mask + 1;
  atomicAdd(&vals[s], w);
  return s;
}

// N(c) of Eq. 2 in the class-synchronous schedule, where the totals are exact: Sigma_c + K_i <= 2m
// (i is not in c) and K_i <= Sigma_d, so with integer weights every factor fits 32 bits.
template <class M>
__device__ __forceinline__ typename M::s_t sweep_score(typename M::h_t kic, typename M::h_t kid, typename M::a_t ki,
                                                       typename M::a_t sc, typename M::a_t sd, typename M::a_t two_m) {
  if constexpr (M::is_fp) return M::score(kic, kid, ki, sc, sd, two_m);
  else return (long long)(int32_t)two_m * (int32_t)(kic - kid) - (long long)(int32_t)ki * (int32_t)(sc - sd + ki);
}

// Order-preserving 64-bit integer of a score, and back.
__device__ __forceinline__ long long score_bits(long long s) { return s; }
__device__ __forceinline__ long long score_bits(double s) {
  const long long b = __double_as_longlong(s);
  return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ void bits_score(long long b, long long& s) { s = b; }
__device__ __forceinline__ void bits_score(long long b, double& s) {
  s = __longlong_as_double(b ^ ((b >> 63) & 0x7fffffffffffffffLL));
}

// Largest score of the warp, ties to the smallest community: three warp reductions (high word, low
// word among its holders, community among theirs).
template <class S>
__device__ __forceinline__ void warp_best(S& s, int32_t& c) {
  const long long b = score_bits(s);
  const int32_t hi = (int32_t)(b >> 32), mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned lo = hi == mh ? (unsigned)b : 0u, ml = __reduce_max_sync(0xffffffffu, lo);
  const unsigned id = hi == mh && lo == ml ? (unsigned)c : 0xffffffffu;
  c = (int32_t)__reduce_min_sync(0xffffffffu, id);
  bits_score(((long long)mh << 32) | ml, s);
}
__device__ __forceinline__ uint32_t warp_total(uint32_t x) { return __reduce_add_sync(0xffffffffu, x); }
__device__ __forceinline__ float warp_total(float x) {
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// State of a step that its parts share.
template <class M>
struct Step {
  const typename M::a_t* sr;  // Sigma: read, and written
  typename M::a_t* sw;
  bool wide;                  // the moves go through mv_from / mv_to
  int nb;                     // move list being filled, its counter
  int* n_moves;
};

// Performs the move of vertex i from d to bc (one thread).
template <class M>
__device__ __forceinline__ void sweep_move(const SweepArgs<M>& a, SweepShared<M>& sh, const Step<M>& sp, int32_t i,
                                           int32_t d, int32_t bc, typename M::a_t ki, typename M::s_t best,
                                           GraphCtl* gcv) {
  a.st.Cp[i] = bc;
  if (sp.wide) {
    a.st.mv_from[i] = d;
    a.st.mv_to[i] = bc;
  } else {
    atomic_add_a(&sp.sw[d], -ki);
    atomic_add_a(&sp.sw[bc], ki);
    const int k = atomicAdd(sp.n_moves, 1);
    if (k < kSwMoves) sh.moves[sp.nb][k] = {d, bc, ki};
    else atomicOr(&a.st.ctrl->error, kErrRange);  // unreachable: such a step is wide
  }
  if (gcv) {
    if (M::is_fp) atomicAdd(&gcv->sum_f, (double)best);
    else atomic_add_u128(&gcv->sum_lo, &gcv->sum_hi, (unsigned long long)best, 0ULL);
  } else if (M::is_fp) {
    atomicAdd(&sh.f, (double)best);
  } else {
    const unsigned long long b = (unsigned long long)best;
    if (atomicAdd(&sh.lo, b) + b < b) atomicAdd(&sh.hi, 1ULL);
  }
  atomicAdd(&sh.mv, 1ULL);
}

// The rows perm[lo, lo + cnt) of one bucket: G threads a row, U arcs a thread (rows hold at most G * U
// arcs), tables of 2^LOG slots.  `rot` shifts which blocks take the first rows.
template <class M, int G, int U, int LOG>
__device__ __forceinline__ void sweep_rows(const SweepArgs<M>& a, SweepShared<M>& sh, const Step<M>& sp, int64_t lo,
                                           int64_t cnt, int64_t rot, typename M::a_t two_m_all) {
  typedef typename M::h_t H;
  typedef typename M::a_t A;
  typedef typename M::s_t S;
  constexpr int GPB = kPersistThreads / G;
  constexpr bool kTable = G > 4;  // four lanes compare their communities directly
  const int gi = threadIdx.x / G, lane = threadIdx.x & (G - 1), warp = threadIdx.x >> 5;
  const int64_t groups = (int64_t)gridDim.x * GPB;
  // few rows: consecutive rows on different blocks; many: on neighbouring groups, which read
  // neighbouring vertices' state
  const int64_t vb = (blockIdx.x + rot) % gridDim.x;
  const int64_t first = cnt > groups ? (int64_t)blockIdx.x * GPB + gi : (int64_t)gi * gridDim.x + vb;
  int32_t* const tk = sh.keys + gi * (kSwSlots / GPB);
  H* const tv = sh.vals + gi * (kSwSlots / GPB);
  static_assert((1 << LOG) <= kSwSlots / GPB, "a group's slice of the table");
  for (int64_t idx = first; idx < cnt; idx += groups) {
    const int32_t i = a.perm[lo + idx];
    const int64_t beg = a.g.rbeg[i];
    const int deg = (int)(a.g.rend[i] - beg);
    const int32_t d = a.st.Cp[i];
    const A ki = a.st.K[i];
    GraphCtl* const gcv = a.st.gc ? a.st.gc + a.st.vg[i] : nullptr;
    bool on = !a.pruning || a.st.flags[i] != 0;
    A two_m = two_m_all;
    if (gcv) {
      on = on && !*(volatile int32_t*)&gcv->done;
      two_m = M::is_fp ? (A)gcv->two_m_f : (A)gcv->two_m_i;
    }
    if (!team_any<G>(on)) continue;
    int32_t jj[U];
    H ww[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
      const int e = lane + u * G;
      jj[u] = e < deg ? a.g.tg[beg + e] : i;
      ww[u] = e < deg ? (H)a.g.w[beg + e] : H(0);
    }
    const A sd = sp.sr[d];
    int32_t cc[U];
#pragma unroll
    for (int u = 0; u < U; u++) cc[u] = jj[u] != i ? a.st.Cp[jj[u]] : d;
    H kid = H(0);
    bool own[U];      // this lane scores community cc[u], whose sum is
    H val[U];
    A sg[U];
    if constexpr (!kTable) {
      const unsigned m = Grp<4>::mask();
      H same = ww[0];
      bool lower = false;
#pragma unroll
      for (int o = 1; o < 4; o++) {
        const int32_t c2 = __shfl_xor_sync(m, cc[0], o);
        const H w2 = __shfl_xor_sync(m, ww[0], o);
        if (c2 == cc[0]) {
          same += w2;
          lower |= (lane ^ o) < lane;
        }
      }
      // padding and i's self-loop carry community d: a lane of d's sums K_i->d without the self-loop
      H mine = jj[0] != i && cc[0] == d ? ww[0] : H(0);
#pragma unroll
      for (int o = 2; o >= 1; o >>= 1) mine += __shfl_xor_sync(m, mine, o);
      kid = mine;
      own[0] = cc[0] != d && !lower;
      val[0] = same;
      sg[0] = own[0] ? sp.sr[cc[0]] : A(0);
    } else {
      const int lg = tbl_log2f_fast(deg, 4, 1, LOG);
      const unsigned size = 1u << lg;
      unsigned sl[U];
      bool ok = true, other[U];
#pragma unroll
      for (int u = 0; u < U; u++) {
        other[u] = cc[u] != d;
        if (jj[u] != i && cc[u] == d) kid += ww[u];
      }
#pragma unroll
      for (int u = 0; u < U; u++) {
        own[u] = false;
        sl[u] = 0;
        if (other[u]) {
          sl[u] = tbl_put(tk, tv, size - 1, 32 - lg, cc[u], ww[u], &own[u]);
          ok &= sl[u] < size;
        }
      }
      if (!ok) atomicOr(&a.st.ctrl->error, kErrTableFull);
#pragma unroll
      for (int u = 0; u < U; u++) sg[u] = own[u] ? sp.sr[cc[u]] : A(0);
      if constexpr (G < 32) {
#pragma unroll
        for (int o = G / 2; o >= 1; o >>= 1) kid += __shfl_xor_sync(Grp<G>::mask(), kid, o);
      } else {
        __syncwarp();
        kid = warp_total(kid);
      }
      if (G > 32 && (lane & 31) == 0) sh.red_h[warp] = kid;
      team_sync<G>();  // every addition is made
      if constexpr (G > 32) kid = warp_total((threadIdx.x & 31) < G / 32 ? sh.red_h[gi * (G / 32) + (threadIdx.x & 31)] : H(0));
#pragma unroll
      for (int u = 0; u < U; u++) {
        val[u] = H(0);
        if (own[u]) {
          val[u] = tv[sl[u]];
          tk[sl[u]] = kEmpty;
          tv[sl[u]] = H(0);
        }
      }
    }
    S best = M::lowest();
    int32_t bc = 0x7fffffff;
#pragma unroll
    for (int u = 0; u < U; u++) {
      if (!own[u]) continue;
      const S sc = sweep_score<M>(val[u], kid, ki, sg[u], sd, two_m);
      if (better(sc, cc[u], best, bc)) { best = sc; bc = cc[u]; }
    }
    if constexpr (G < 32) {
      group_argmax<G>(best, bc, (S*)nullptr, (int32_t*)nullptr);
    } else {
      __syncwarp();
      warp_best(best, bc);
    }
    if constexpr (G > 32) {
      if ((threadIdx.x & 31) == 0) {
        sh.red_s[warp] = best;
        sh.red_c[warp] = bc;
      }
      team_sync<G>();
      const bool in = (threadIdx.x & 31) < G / 32;
      best = in ? sh.red_s[gi * (G / 32) + (threadIdx.x & 31)] : M::lowest();
      bc = in ? sh.red_c[gi * (G / 32) + (threadIdx.x & 31)] : 0x7fffffff;
      warp_best(best, bc);
    } else {
      team_sync<G>();  // the table is empty again
    }
    if (a.pruning && lane == 0) a.st.flags[i] = 0;
    if (bc != 0x7fffffff && best > S(0)) {
      if (lane == 0) sweep_move(a, sh, sp, i, d, bc, ki, best, gcv);
      if (a.pruning) {
#pragma unroll
        for (int u = 0; u < U; u++)
          if (jj[u] != i) a.st.flags[jj[u]] = 1;
      }
    }
  }
}

// The class's giants of at most kSwLongest arcs, a block each: eight arcs a thread in two steps, the
// slots a thread claimed as 16-bit halves.
template <class M>
__device__ __forceinline__ void sweep_long_rows(const SweepArgs<M>& a, SweepShared<M>& sh, const Step<M>& sp,
                                                const int32_t* list, int64_t k0, int64_t k1,
                                                typename M::a_t two_m_all) {
  typedef typename M::h_t H;
  typedef typename M::a_t A;
  typedef typename M::s_t S;
  constexpr int G = kPersistThreads, U = 4, LOG = 14;
  static_assert(2 * G * U == kSwLongest && (1 << LOG) == kSwSlots, "two steps, the whole table");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int64_t k = k0 + blockIdx.x; k < k1; k += gridDim.x) {
    const int32_t i = list[k];
    const int64_t beg = a.g.rbeg[i], end = a.g.rend[i];
    if (end - beg > kSwLongest) continue;
    const int deg = (int)(end - beg);
    const int32_t d = a.st.Cp[i];
    const A ki = a.st.K[i];
    GraphCtl* const gcv = a.st.gc ? a.st.gc + a.st.vg[i] : nullptr;
    bool on = !a.pruning || a.st.flags[i] != 0;
    A two_m = two_m_all;
    if (gcv) {
      on = on && !*(volatile int32_t*)&gcv->done;
      two_m = M::is_fp ? (A)gcv->two_m_f : (A)gcv->two_m_i;
    }
    if (!team_any<G>(on)) continue;
    const A sd = sp.sr[d];
    H kid = H(0);
    unsigned claim[U];  // step 0's slot in the low half, step 1's in the high half
    bool ok = true;
#pragma unroll
    for (int u = 0; u < U; u++) claim[u] = 0xffffffffu;
#pragma unroll
    for (int h = 0; h < 2; h++) {
      int32_t jj[U], cc[U];
      H ww[U];
#pragma unroll
      for (int u = 0; u < U; u++) {
        const int e = (int)threadIdx.x + (h * U + u) * G;
        jj[u] = e < deg ? a.g.tg[beg + e] : i;
        ww[u] = e < deg ? (H)a.g.w[beg + e] : H(0);
      }
#pragma unroll
      for (int u = 0; u < U; u++) cc[u] = jj[u] != i ? a.st.Cp[jj[u]] : d;
#pragma unroll
      for (int u = 0; u < U; u++) {
        if (jj[u] != i && cc[u] == d) kid += ww[u];
        if (cc[u] != d) {
          bool own;
          const unsigned sl = tbl_put(sh.keys, sh.vals, kSwSlots - 1, 32 - LOG, cc[u], ww[u], &own);
          if (own) claim[u] = h ? ((claim[u] & 0xffffu) | (sl << 16)) : ((claim[u] & 0xffff0000u) | sl);
          ok &= sl < kSwSlots;
        }
      }
    }
    if (!ok) atomicOr(&a.st.ctrl->error, kErrTableFull);
    __syncwarp();
    kid = warp_total(kid);
    if (lane == 0) sh.red_h[warp] = kid;
    __syncthreads();
    kid = warp_total(sh.red_h[lane]);
    S best = M::lowest();
    int32_t bc = 0x7fffffff;
#pragma unroll
    for (int h = 0; h < 2; h++) {
      int32_t key[U];
      H val[U];
      A sg[U];
#pragma unroll
      for (int u = 0; u < U; u++) {
        const unsigned sl = h ? claim[u] >> 16 : claim[u] & 0xffffu;
        key[u] = kEmpty;
        val[u] = H(0);
        if (sl != 0xffffu) {
          key[u] = sh.keys[sl];
          val[u] = sh.vals[sl];
          sh.keys[sl] = kEmpty;
          sh.vals[sl] = H(0);
        }
      }
#pragma unroll
      for (int u = 0; u < U; u++) sg[u] = key[u] != kEmpty ? sp.sr[key[u]] : A(0);
#pragma unroll
      for (int u = 0; u < U; u++) {
        if (key[u] == kEmpty) continue;
        const S sc = sweep_score<M>(val[u], kid, ki, sg[u], sd, two_m);
        if (better(sc, key[u], best, bc)) { best = sc; bc = key[u]; }
      }
    }
    __syncwarp();
    warp_best(best, bc);
    if (lane == 0) {
      sh.red_s[warp] = best;
      sh.red_c[warp] = bc;
    }
    __syncthreads();
    best = sh.red_s[lane];
    bc = sh.red_c[lane];
    warp_best(best, bc);
    if (a.pruning && threadIdx.x == 0) a.st.flags[i] = 0;
    if (bc != 0x7fffffff && best > S(0)) {
      if (threadIdx.x == 0) sweep_move(a, sh, sp, i, d, bc, ki, best, gcv);
      if (a.pruning)
        for (int e = threadIdx.x; e < deg; e += G) {
          const int32_t j = a.g.tg[beg + e];
          if (j != i) a.st.flags[j] = 1;
        }
    }
  }
}

// Arcs of the class's flagged giants into their tables: a warp takes 32 * U arcs.
template <class M, int U>
__device__ __forceinline__ void sweep_giant_insert(const SweepArgs<M>& a, const GiantAct& ga, const int32_t* list,
                                                   int64_t k0, int64_t k1) {
  typedef typename M::h_t H;
  constexpr int kPieces = kLmChunk / (32 * U);
  const GiantPlan& p = a.gp;
  const int lane = threadIdx.x & 31;
  const int64_t q0 = p.chunk_off[k0], np = (p.chunk_off[k1] - q0) * kPieces;
  bool ok = true;
  for (int64_t t = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x; t < np; t += (int64_t)gridDim.x * kSwWarps) {
    const int64_t q = q0 + t / kPieces, k = p.cowner[q];
    const int32_t i = list[k];
    const int64_t c0 = p.chunk_off[k], beg = a.g.rbeg[i], e1 = a.g.rend[i];
    const bool act = giant_active(ga, p, k, i) && e1 - beg > kSwLongest;
    if (q == c0 && t % kPieces == 0 && lane == 0) p.active[k] = act ? 1 : 0;  // for the later parts of the step
    if (!act) continue;
    const int32_t d = a.st.Cp[i];
    const int64_t ts = p.tab_off[k + 1] - p.tab_off[k];
    const int64_t off = p.tab_off[k] - p.tab_off[k0];  // the step's tables from the pool's start
    const int lg = 63 - __clzll(ts);
    int32_t* kv = p.slots + 2 * off;
    const int64_t e0 = beg + (q - c0) * kLmChunk + (t % kPieces) * (32 * U) + lane;
    int32_t jj[U];
    H ww[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
      jj[u] = e0 + u * 32 < e1 ? a.g.tg[e0 + u * 32] : i;
      ww[u] = e0 + u * 32 < e1 ? (H)a.g.w[e0 + u * 32] : H(0);
    }
    int32_t cc[U], seen[U];
    unsigned home[U];
    bool other[U];
    H kid = H(0);
#pragma unroll
    for (int u = 0; u < U; u++) cc[u] = jj[u] != i ? a.st.Cp[jj[u]] : d;
#pragma unroll
    for (int u = 0; u < U; u++) {
      other[u] = cc[u] != d;
      if (jj[u] != i && cc[u] == d) kid += ww[u];
    }
#pragma unroll
    for (int u = 0; u < U; u++) {
      home[u] = tbl_home(cc[u], 32 - lg);
      seen[u] = other[u] ? *((volatile int32_t*)&kv[2 * (size_t)home[u]]) : 0;
    }
#pragma unroll
    for (int u = 0; u < U; u++) {
      if (other[u]) ok &= tbl_add_mark_at(kv, (unsigned)ts, cc[u], ww[u], p.bits, off, home[u], seen[u]);
    }
    __syncwarp();
    kid = warp_total(kid);
    if (lane == 0 && kid != H(0)) atomicAdd(reinterpret_cast<H*>(p.kid) + k, kid);
  }
  if (!ok) atomicOr(&a.st.ctrl->error, kErrTableFull);
}

// Best candidate of every 1024-slot range of the class's flagged giants: 128 threads a range, eight
// bitmap words a warp, a lane per slot of a word (coalesced).  Slots and bits are cleared.
template <class M>
__device__ __forceinline__ void sweep_giant_scan(const SweepArgs<M>& a, SweepShared<M>& sh, const Step<M>& sp,
                                                 const int32_t* list, int64_t k0, int64_t k1,
                                                 typename M::a_t two_m_all) {
  typedef typename M::h_t H;
  typedef typename M::a_t A;
  typedef typename M::s_t S;
  constexpr int W = 8;
  const GiantPlan& p = a.gp;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, team = threadIdx.x >> 7;
  const int64_t r0 = p.slice_off[k0], r1 = p.slice_off[k1];
  for (int64_t q = r0 + (int64_t)team * gridDim.x + blockIdx.x; q < r1; q += (int64_t)gridDim.x * (kPersistThreads / 128)) {
    const int64_t k = p.sowner[q];
    if (!p.active[k]) continue;  // uniform over the team
    const int32_t i = list[k];
    const int32_t d = a.st.Cp[i];
    const int64_t off = p.tab_off[k] - p.tab_off[k0], ts = p.tab_off[k + 1] - p.tab_off[k];
    const H kid = reinterpret_cast<const H*>(p.kid)[k];
    const A ki = a.st.K[i], sd = sp.sr[d];
    const A two_m = a.st.gc ? (M::is_fp ? (A)a.st.gc[a.st.vg[i]].two_m_f : (A)a.st.gc[a.st.vg[i]].two_m_i) : two_m_all;
    const int64_t sb = ((q - p.slice_off[k]) << kRangeLog) + (warp & 3) * (32 * W);
    int2* kv = reinterpret_cast<int2*>(p.slots) + off + sb;
    unsigned* wp = p.bits + ((off + sb) >> 5);
    const int nwords = sb >= ts ? 0 : (int)(ts - sb < 32 * W ? (ts - sb) >> 5 : W);
    const unsigned word = lane < nwords ? wp[lane] : 0u;
    if (word) wp[lane] = 0u;
    int2 e[W];
#pragma unroll
    for (int x = 0; x < W; x++) {
      const unsigned bits = __shfl_sync(0xffffffffu, word, x);
      e[x] = (bits >> lane) & 1u ? kv[x * 32 + lane] : make_int2(kEmpty, 0);
    }
    A sg[W];
#pragma unroll
    for (int x = 0; x < W; x++) sg[x] = e[x].x != kEmpty ? sp.sr[e[x].x] : A(0);
    S best = M::lowest();
    int32_t bc = 0x7fffffff;
#pragma unroll
    for (int x = 0; x < W; x++) {
      if (e[x].x == kEmpty) continue;
      kv[x * 32 + lane] = make_int2(kEmpty, 0);
      const S sc = sweep_score<M>(int_as_h<H>(e[x].y), kid, ki, sg[x], sd, two_m);
      if (better(sc, e[x].x, best, bc)) { best = sc; bc = e[x].x; }
    }
    __syncwarp();
    warp_best(best, bc);
    if (lane == 0) {
      sh.red_s[warp] = best;
      sh.red_c[warp] = bc;
    }
    team_sync<128>();
    if ((threadIdx.x & 127) == 0) {
      for (int w = 1; w < 4; w++)
        if (better(sh.red_s[warp + w], sh.red_c[warp + w], best, bc)) { best = sh.red_s[warp + w]; bc = sh.red_c[warp + w]; }
      reinterpret_cast<S*>(p.part_s)[q] = best;
      p.part_c[q] = bc;
    }
    team_sync<128>();
  }
}

// Moves the class's giants whose best candidate gains and marks their neighbours: every warp that
// takes arcs of a giant reduces its ranges' candidates, the one with its first arcs moves it.
template <class M>
__device__ __forceinline__ void sweep_giant_decide(const SweepArgs<M>& a, SweepShared<M>& sh, const Step<M>& sp,
                                                   const int32_t* list, int64_t k0, int64_t k1) {
  typedef typename M::s_t S;
  constexpr int U = 4, kPieces = kLmChunk / (32 * U);
  const GiantPlan& p = a.gp;
  const int lane = threadIdx.x & 31;
  const int64_t q0 = p.chunk_off[k0], np = (p.chunk_off[k1] - q0) * kPieces;
  for (int64_t t = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x; t < np; t += (int64_t)gridDim.x * kSwWarps) {
    const int64_t q = q0 + t / kPieces, k = p.cowner[q];
    if (!p.active[k]) continue;
    const int32_t i = list[k];
    const int64_t c0 = p.chunk_off[k];
    const int64_t e0 = a.g.rbeg[i] + (q - c0) * kLmChunk + (t % kPieces) * (32 * U) + lane, e1 = a.g.rend[i];
    int32_t jj[U];
#pragma unroll
    for (int u = 0; u < U; u++) jj[u] = a.pruning && e0 + u * 32 < e1 ? a.g.tg[e0 + u * 32] : i;
    S best = M::lowest();
    int32_t bc = 0x7fffffff;
    for (int64_t x = p.slice_off[k] + lane; x < p.slice_off[k + 1]; x += 32) {
      const S s = reinterpret_cast<const S*>(p.part_s)[x];
      const int32_t c = p.part_c[x];
      if (better(s, c, best, bc)) { best = s; bc = c; }
    }
    __syncwarp();
    warp_best(best, bc);
    const bool mv = bc != 0x7fffffff && best > S(0);
    if (q == c0 && t % kPieces == 0 && lane == 0) {
      reinterpret_cast<uint32_t*>(p.kid)[k] = 0u;  // for the next use of the plan (0u is also 0.0f)
      if (a.pruning) a.st.flags[i] = 0;
      if (mv) sweep_move(a, sh, sp, i, a.st.Cp[i], bc, a.st.K[i], best, a.st.gc ? a.st.gc + a.st.vg[i] : nullptr);
    }
    if (mv) {
#pragma unroll
      for (int u = 0; u < U; u++)
        if (jj[u] != i) a.st.flags[jj[u]] = 1;
    }
  }
}

// Algorithm 2's tolerance test: 2 sum N <= tau (2m)^2 (the arithmetic of lm_finish).
template <bool FP>
__device__ __forceinline__ bool sweep_converged(unsigned long long lo, unsigned long long hi, double f, double tau,
                                                long long two_m_i, double two_m_f) {
  if (FP) return __dmul_rn(2.0, f) <= __dmul_rn(tau, __dmul_rn(two_m_f, two_m_f));
  const double t = __ll2double_rn(two_m_i);
  return u128_to_double_rn((hi << 1) | (lo >> 63), lo << 1) <= __dmul_rn(tau, __dmul_rn(t, t));
}

template <class M, int SC>
__global__ void __launch_bounds__(kPersistThreads, 1) lm_sweep(SweepArgs<M> a, PersistBar bar) {
  typedef typename M::a_t A;
  typedef typename M::h_t H;
  extern __shared__ __align__(16) unsigned char sw_dyn[];
  SweepShared<M>& sh = *reinterpret_cast<SweepShared<M>*>(sw_dyn);
  Ctrl* const ctrl = a.st.ctrl;
  if (*(volatile int32_t*)&ctrl->done) return;
  const int tid = threadIdx.x;
  for (int t = tid; t < kSwSlots; t += kPersistThreads) { sh.keys[t] = kEmpty; sh.vals[t] = H(0); }
  if (tid < kStepWords) sh.rec[0][tid] = a.recs[tid];
  if (tid < 3) sh.n_moves[tid] = 0;
  if (tid == 0) { sh.lo = sh.hi = sh.mv = 0; sh.f = 0.0; sh.done = sh.act = 0; }
  for (int64_t c = (int64_t)blockIdx.x * kPersistThreads + tid; c < a.n_sig; c += (int64_t)gridDim.x * kPersistThreads)
    a.sig2[c] = a.st.Sig[c];
  const A two_m = M::is_fp ? (A)ctrl->two_m_f : (A)ctrl->two_m_i;
  GiantAct ga;
  ga.snap = 0;
  ga.pruning = a.pruning;
  ga.flags = a.st.flags;
  ga.gc = a.st.gc;
  ga.vg = a.st.vg;
  unsigned long long sum;
  auto none = []() { return 0ULL; };
  if (!scope_barrier<SC>(bar, ctrl, &sum, none)) return;
  A* const sig[2] = {a.st.Sig, a.sig2};
  int par = 0;           // Sigma copy that the step reads
  unsigned n = 0;        // steps taken: the moves of step n are in list n % 2, their number in n_moves[n % 3]
  int it = 0;            // iterations finished
  while (true) {
    for (int s = 0; s < a.nsteps; s++, n++) {
      const int64_t* rec = sh.rec[n & 1];
      if (tid >= kPersistThreads - kStepWords) {  // the next step's record, for after the barrier
        const int x = tid - (kPersistThreads - kStepWords);
        sh.rec[(n + 1) & 1][x] = a.recs[(int64_t)(s + 1 < a.nsteps ? s + 1 : 0) * kStepWords + x];
      }
      Step<M> sp;
      sp.sr = sig[par];
      sp.sw = sig[par ^ 1];
      sp.wide = a.all_wide || rec[kStepWide] != 0;
      sp.nb = n & 1;
      sp.n_moves = &sh.n_moves[n % 3];
      const int32_t* list = a.glist + rec[kStepGiant];
      const int64_t k0 = rec[kStepGiant + 1], k1 = rec[kStepGiant + 2];
      bool act = false;
      for (int64_t k = k0 + tid; k < k1; k += kPersistThreads) {
        const int32_t v = list[k];
        act |= a.g.rend[v] - a.g.rbeg[v] > kSwLongest && giant_active(ga, a.gp, k, v);
      }
      // the last step's moves on the copy that lacks them
      {
        const SweepMove<M>* mv = sh.moves[(n + 1) & 1];
        const int nm = min(sh.n_moves[(n + 2) % 3], kSwMoves);
        for (int t = tid; t < nm; t += kPersistThreads) {
          atomic_add_a(&sp.sw[mv[t].from], -mv[t].k);
          atomic_add_a(&sp.sw[mv[t].to], mv[t].k);
        }
      }
      if (k1 > k0) {
        const int64_t arcs = (a.gp.chunk_off[k1] - a.gp.chunk_off[k0]) * kLmChunk;
        if (arcs <= (int64_t)gridDim.x * kPersistThreads) sweep_giant_insert<M, 1>(a, ga, list, k0, k1);
        else sweep_giant_insert<M, 4>(a, ga, list, k0, k1);
      }
      sweep_long_rows<M>(a, sh, sp, list, k0, k1, two_m);
      // long rows first; each bucket's rows start on the blocks after the last bucket's
      if (rec[11] > 0) sweep_rows<M, 1024, 4, 14>(a, sh, sp, rec[10], rec[11], gridDim.x - (k1 - k0) % gridDim.x, two_m);
      if (rec[9] > 0) sweep_rows<M, 512, 4, 13>(a, sh, sp, rec[8], rec[9], gridDim.x - (k1 - k0 + rec[11]) % gridDim.x, two_m);
      if (rec[7] > 0) sweep_rows<M, 128, 4, 11>(a, sh, sp, rec[6], rec[7], gridDim.x - (k1 - k0 + rec[11] + rec[9]) % gridDim.x, two_m);
      if (rec[5] > 0) sweep_rows<M, 32, 4, 9>(a, sh, sp, rec[4], rec[5], gridDim.x - (k1 - k0 + rec[11] + rec[9] + rec[7]) % gridDim.x, two_m);
      if (rec[3] > 0) sweep_rows<M, 8, 2, 6>(a, sh, sp, rec[2], rec[3], 0, two_m);
      if (rec[1] > 0) sweep_rows<M, 4, 1, 3>(a, sh, sp, rec[0], rec[1], 0, two_m);
      const bool last = s + 1 == a.nsteps && a.whole && !a.st.gc;
      auto flush = [&]() {  // thread 0: the block's sums of the iteration travel with the last step's barrier
        if (!last) return;
        unsigned long long* t = a.state + kSwSums + 4 * (it % 3);
        if (sh.mv) {
          atomicAdd(&t[3], sh.mv);
          if (M::is_fp) atomicAdd(reinterpret_cast<double*>(&t[2]), sh.f);
          else atomic_add_u128(&t[0], &t[1], sh.lo, sh.hi);
        }
        sh.lo = sh.hi = sh.mv = 0;
        sh.f = 0.0;
      };
      if (act) sh.act = 1;
      bool ok = scope_barrier<SC>(bar, ctrl, &sum, [&]() {
        flush();
        const unsigned long long x = (unsigned long long)sh.act;
        sh.act = 0;
        return x;
      });
      if (!ok) return;
      if (sum & kBarSum) {  // some giant of the class is flagged
        sweep_giant_scan<M>(a, sh, sp, list, k0, k1, two_m);
        if (!scope_barrier<SC>(bar, ctrl, &sum, none)) return;
        sweep_giant_decide<M>(a, sh, sp, list, k0, k1);
        ok = scope_barrier<SC>(bar, ctrl, &sum, [&]() {
          flush();
          return 0ULL;
        });
        if (!ok) return;
      }
      if (sp.wide) {
        const int64_t v0 = rec[kStepApply], v1 = v0 + rec[kStepApply + 1];
        for (int64_t v = v0 + (int64_t)blockIdx.x * kPersistThreads + tid; v < v1; v += (int64_t)gridDim.x * kPersistThreads) {
          const int32_t i = a.perm[v], to = a.st.mv_to[i];
          if (to < 0) continue;
          const int32_t from = a.st.mv_from[i];
          const A ki = a.st.K[i];
          atomic_add_a(&sp.sw[from], -ki);
          atomic_add_a(&sp.sw[to], ki);
          atomic_add_a(&sig[par][from], -ki);
          atomic_add_a(&sig[par][to], ki);
          a.st.mv_to[i] = -1;
        }
        if (!scope_barrier<SC>(bar, ctrl, &sum, none)) return;
      }
      par ^= 1;
      if (tid == 0) sh.n_moves[(n + 2) % 3] = 0;  // read in this step, filled in the step after next
    }
    if (!a.whole) break;
    it++;
    bool stop;
    if (a.st.gc) {
      // per graph; the graphs left come with the barrier
      const double tau = ctrl->tau;
      int left = 0;
      for (int g = blockIdx.x * kPersistThreads + tid; g < a.n_graphs; g += gridDim.x * kPersistThreads) {
        GraphCtl& c = a.st.gc[g];
        if (c.done) continue;
        c.iterations = it;
        const bool conv = sweep_converged<M::is_fp>(c.sum_lo, c.sum_hi, c.sum_f, tau, c.two_m_i, c.two_m_f);
        c.sum_lo = c.sum_hi = 0;
        c.sum_f = 0.0;
        if (conv || it >= ctrl->max_iterations) c.done = 1;
        else left++;
      }
      if (left) atomicAdd(&sh.done, left);
      const bool ok = scope_barrier<SC>(bar, ctrl, &sum, [&]() {
        const unsigned long long x = (unsigned long long)sh.done;
        sh.done = 0;
        return x;
      });
      if (!ok) return;
      stop = (sum & kBarSum) == 0;
    } else {
      if (tid == 0) {
        const volatile unsigned long long* t = a.state + kSwSums + 4 * ((it - 1) % 3);
        const unsigned long long lo = t[0], hi = t[1], f = t[2];
        sh.done = sweep_converged<M::is_fp>(lo, hi, __longlong_as_double((long long)f), ctrl->tau, ctrl->two_m_i,
                                            ctrl->two_m_f) || it >= ctrl->max_iterations;
        if (blockIdx.x == 0) {
          ctrl->moves_pass += t[3];
          unsigned long long* z = a.state + kSwSums + 4 * ((it + 1) % 3);  // last read before this iteration
          z[0] = z[1] = z[2] = z[3] = 0;
        }
      }
      __syncthreads();
      stop = sh.done != 0;
    }
    if (stop) break;
  }
  // both copies hold every move in the end
  {
    const SweepMove<M>* mv = sh.moves[(n + 1) & 1];
    const int nm = min(sh.n_moves[(n + 2) % 3], kSwMoves);
    A* const s = sig[par ^ 1];
    for (int t = tid; t < nm; t += kPersistThreads) {
      atomic_add_a(&s[mv[t].from], -mv[t].k);
      atomic_add_a(&s[mv[t].to], mv[t].k);
    }
  }
  __syncthreads();
  if (tid == 0) {
    if (a.whole && blockIdx.x == 0) {
      ctrl->iterations = it;
      ctrl->done = 1;
    }
    if ((!a.whole || a.st.gc) && sh.mv) {  // sums left for the kernel that finishes the iteration
      if (a.whole) {
        atomicAdd(&ctrl->moves_pass, sh.mv);
      } else {
        atomicAdd(&ctrl->moves, sh.mv);
        if (M::is_fp) atomicAdd(&ctrl->sum_f, sh.f);
        else atomic_add_u128(&ctrl->sum_lo, &ctrl->sum_hi, sh.lo, sh.hi);
      }
    }
  }
}

template <class M>
cudaError_t move_sweep(Ctx& c, const SweepPlan& sw, const GraphView<typename M::w_t>& g, const PassState<M>& st,
                       const int32_t* perm, const int32_t* glist, const GiantPlan& gp, bool pruning, int32_t n_graphs) {
  SweepArgs<M> a;
  a.g = g; a.st = st; a.perm = perm; a.glist = glist; a.gp = gp;
  a.sig2 = reinterpret_cast<typename M::a_t*>(sw.sig2);
  a.n_sig = g.n;
  a.recs = sw.recs;
  a.nsteps = sw.nsteps;
  a.whole = sw.whole ? 1 : 0;
  a.pruning = pruning ? 1 : 0;
  a.n_graphs = n_graphs;
  a.all_wide = 0;
  a.state = sw.state;
  cudaError_t e = cudaMemsetAsync(sw.state, 0, kSwWords * sizeof(unsigned long long), c.s);
  if (e != cudaSuccess) return e;
  const PersistBar bar{sw.state + kSwBar, c.wait_spins > 0 ? c.wait_spins : kBarrierPolls, 0};
  const Scope sc = c.wait_spins > 0 ? kGrid : (Scope)sw.scope;
  constexpr size_t smem = sizeof(SweepShared<M>);
  if (sc == kCta) e = scope_launch(sc, c, lm_sweep<M, kCta>, smem, a, bar);
  else if (sc == kCluster) e = scope_launch(sc, c, lm_sweep<M, kCluster>, smem, a, bar);
  else e = scope_launch(sc, c, lm_sweep<M, kGrid>, smem, a, bar);
  if (e != cudaSuccess && sc != kCta) {  // the scope cannot be launched here: one block can
    cudaGetLastError();
    a.all_wide = 1;
    e = scope_launch(kCta, c, lm_sweep<M, kCta>, smem, a, bar);
  }
  c.launches++;
  return e;
}

template cudaError_t move_sweep<IntMode>(Ctx&, const SweepPlan&, const GraphView<int32_t>&, const PassState<IntMode>&,
                                         const int32_t*, const int32_t*, const GiantPlan&, bool, int32_t);
template cudaError_t move_sweep<FpMode>(Ctx&, const SweepPlan&, const GraphView<float>&, const PassState<FpMode>&,
                                        const int32_t*, const int32_t*, const GiantPlan&, bool, int32_t);

}  // namespace lv
