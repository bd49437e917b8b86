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
//   * a row of every bucket fits its group in one step (4 lanes to 4 arcs, no table: lanes compare their
//     communities by shuffles; 8 lanes to 16, a warp to 128, 64 threads to 512, 256 to 2048, 512 to 4096,
//     and to 8192 in two steps), so its targets are still in registers when a move marks its neighbours;
//     the tables of all group sizes are slices of one 16384-slot table;
//   * the lane that claims a slot scores and clears it: its Sigma_c load is issued at the claim;
//   * with several blocks a step gives every block one kind of row, in numbers that let the kinds finish
//     together, and what a step cannot change of its rows (head, arcs) is loaded during the barrier
//     before it: after the barrier come C'[j], Sigma_c and the table, two trips to L2 instead of five;
//   * Sigma is kept twice.  A step reads one copy and adds its moves to the other; the next step
//     swaps them and first repeats those moves (kept in shared memory) on the copy that lacks them.
//     So a step needs no second barrier between deciding and applying.  A step with more vertices
//     than a block can keep decides, waits, and applies to both copies;
//   * giant rows over 8192 arcs: arcs insert into the shared pool by the warp, a barrier, 128 threads
//     score 1024 slots, a barrier, and every warp that marks a giant's arcs reduces the giant's
//     candidates itself; scoring and deciding are skipped when no giant of the class is flagged;
//   * the tolerance test is made by every block from sums that come with the last step's barrier.
// R-MAT 22, passes 0 and 1 (350 and 382 classes, 2 and 4 iterations): 21.2 and 38.5 ms (per-class
// launches 33.0 and 54.0); R-MAT 20: 9.8 and 23.2 (19.1 and 39.5); SBM 10k, three passes: 0.72, 0.67 and
// 0.26 (1.2, 2.0 and 0.97); 24M-vertex grid, last two passes: 4.6 and 3.5 (12.2 and 12.2).
// Integer results are those of the separate kernels bit for bit (exact sums, ties by id).
#include "giant.cuh"
#include "persist.cuh"

namespace lv {

// Table slots of a block, divided among its groups: four per arc of the longest row of a bucket (half
// full, a 4096-arc row's insertion takes 11,000 cycles of probing against 4,000), two per arc of the
// longest row a block takes.
constexpr int kSwSlots = 16384;
constexpr int kSwMoves = kSweepMoves;
// Threads of a block.  A phase with rows over 512 arcs takes 512 of 128 registers: with 1024 of 64 the
// step's state spills, and after a barrier, which empties L1, every reload is a trip to L2 (R-MAT 20,
// pass 1: 26.6 ms with 1024 threads, 22.6 with 512).  One without them needs less state a thread and
// more rows in flight: 1024.
constexpr int kSwThreads = 512;
constexpr int kSwWarps = kSwThreads / 32;
constexpr int kSwLowThreads = 1024;

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
  int all_wide;               // 1: the launch has fewer blocks than the records were made for: the blocks'
                              // kinds of rows and move counts in them do not hold
  GiantPlan gp;
  unsigned long long* state;  // kSw* below, zeroed before the launch
};
// 3 barrier words, then 3 rotating sums of an iteration {lo, hi, fp, moves}
enum { kSwBar = 0, kSwSums = 4, kSwWords = kSwSums + 12 };
static_assert(kSwWords <= kSweepStateWords, "state block");

constexpr int kSwPool = 32;  // pool giants taken at once: one a lane

struct GiantDesc {
  int64_t beg;     // row start
  int64_t tab;     // first slot of its table, the batch's tables from the pool's start
  int64_t part;    // first of its range results
  int64_t k;       // index in the plan
  int32_t i, deg, lg, pad;
};

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
  int64_t rec[4][kStepWords];     // records of the last and the next three steps
  GiantDesc gd[3][kSwPool];       // pool giants of the last and the next two steps,
  GiantDesc gdx[kSwPool];         // of a further batch of a step
  typename M::s_t red_s[32];
  int32_t red_c[32];
  typename M::h_t red_h[32];
  unsigned long long lo, hi, mv;  // this block's sums of the iteration
  double f;
  int done;
  typename M::a_t two_m;          // of a single graph
};

// A group of G threads: lanes of a warp, or whole warps that meet at a named barrier (64-thread groups
// 1-8, 128-thread groups 1-8, 256-thread groups 9-10, the block 0).
template <int G, int T>
__device__ __forceinline__ void team_sync() {
  if constexpr (G < 32) __syncwarp(Grp<G>::mask());
  else if constexpr (G == 32) __syncwarp();
  else if constexpr (G == T) __syncthreads();
  else {
    const int id = (G <= 128 ? 1 : 9) + (int)threadIdx.x / G;
    asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(G) : "memory");
  }
}

// Whether any thread of the group says so: the same answer on all of them, whatever changes meanwhile.
template <int G, int T>
__device__ __forceinline__ bool team_any(bool p) {
  if constexpr (G <= 32) return __any_sync(Grp<G>::mask(), p);
  else if constexpr (G == T) return __syncthreads_or(p ? 1 : 0) != 0;
  else {
    const int id = (G <= 128 ? 1 : 9) + (int)threadIdx.x / G;
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

// What a row needs that no step changes, loaded ahead: its head, then this thread's arcs.
template <class M>
struct Head {
  int32_t i;                 // vertex, -1: none
  int deg;
  int64_t beg;
  int32_t at;                // its graph (batch)
  int on;                    // flagged (only ever set, except by its own step)
  typename M::a_t ki;
};
template <class M, int N>
struct Arcs {
  int32_t jj[N];             // targets (the row's vertex past its end) and weights
  typename M::h_t ww[N];
};

template <class M>
__device__ __forceinline__ void load_head(const SweepArgs<M>& a, int32_t i, Head<M>& h) {
  h.i = i;
  h.beg = a.g.rbeg[i];
  h.deg = (int)(a.g.rend[i] - h.beg);
  h.ki = a.st.K[i];
  h.at = a.st.gc ? a.st.vg[i] : 0;
  h.on = !a.pruning || a.st.flags[i] != 0;
}
// Arcs [beg + lane + u * G], u < U, of a row of `deg` arcs from beg.
template <class M, int N>
__device__ __forceinline__ void load_arcs(const SweepArgs<M>& a, int32_t i, int64_t beg, int deg, int lane, int G, int U,
                                          Arcs<M, N>& r) {
#pragma unroll
  for (int u = 0; u < N; u++) {
    const int e = lane + u * G;
    const bool in = u < U && e < deg;
    r.jj[u] = in ? a.g.tg[beg + e] : i;
    r.ww[u] = in ? (typename M::h_t)a.g.w[beg + e] : typename M::h_t(0);
  }
}

// Decides row h with this thread's arcs r (if `loaded`): G threads a row, U arcs a thread, R rounds of
// them (the later rounds' arcs are loaded here), tables of 2^LOG slots.  `sure`: h.on was read in this
// step, in which nothing else marks the class's rows.
template <class M, class R_, int T, int N>
__device__ __forceinline__ void sweep_row(const SweepArgs<M>& a, SweepShared<M>& sh, const Step<M>& sp, const Head<M>& h,
                                          Arcs<M, N>& r, bool loaded, bool sure) {
  constexpr int G = R_::G, U = R_::U, LOG = R_::LOG, R = R_::R;
  typedef typename M::h_t H;
  typedef typename M::a_t A;
  typedef typename M::s_t S;
  constexpr int GPB = T / G;
  const int gi = threadIdx.x / G, lane = threadIdx.x & (G - 1), warp = threadIdx.x >> 5;
  int32_t* const tk = sh.keys + gi * (kSwSlots / GPB);
  H* const tv = sh.vals + gi * (kSwSlots / GPB);
  static_assert((1 << LOG) <= kSwSlots / GPB, "a group's slice of the table");
  if (sure && !team_any<G, T>(h.on != 0)) return;
  const int32_t i = h.i, d = a.st.Cp[i];
  const A ki = h.ki;
  int32_t cc[U];
  if (loaded) {
#pragma unroll
    for (int u = 0; u < U; u++) cc[u] = a.st.Cp[r.jj[u]];
  }
  GraphCtl* const gcv = a.st.gc ? a.st.gc + h.at : nullptr;
  bool on = h.on || (!sure && a.st.flags[i] != 0);
  A two_m = *(volatile A*)&sh.two_m;
  if (gcv) {
    on = on && !*(volatile int32_t*)&gcv->done;
    two_m = M::is_fp ? (A)gcv->two_m_f : (A)gcv->two_m_i;
  }
  if (!team_any<G, T>(on)) return;
  const A sd = sp.sr[d];
  if (!loaded) {
    load_arcs(a, i, h.beg, h.deg, lane, G, U, r);
#pragma unroll
    for (int u = 0; u < U; u++) cc[u] = a.st.Cp[r.jj[u]];
  }
  H kid = H(0);
  S best = M::lowest();
  int32_t bc = 0x7fffffff;
  if constexpr (G == 4 && U == 1) {  // four arcs: the lanes compare their communities
    const unsigned m = Grp<4>::mask();
    if (r.jj[0] == i) cc[0] = d;  // padding and i's self-loop
    H same = r.ww[0];
    bool lower = false;
#pragma unroll
    for (int o = 1; o < 4; o++) {
      const int32_t c2 = __shfl_xor_sync(m, cc[0], o);
      const H w2 = __shfl_xor_sync(m, r.ww[0], o);
      if (c2 == cc[0]) {
        same += w2;
        lower |= (lane ^ o) < lane;
      }
    }
    const bool own = cc[0] != d && !lower;
    const A sg = own ? sp.sr[cc[0]] : A(0);
    kid = r.jj[0] != i && cc[0] == d ? r.ww[0] : H(0);
#pragma unroll
    for (int o = 2; o >= 1; o >>= 1) kid += __shfl_xor_sync(m, kid, o);
    if (own) {
      best = sweep_score<M>(same, kid, ki, sg, sd, two_m);
      bc = cc[0];
    }
    group_argmax<4>(best, bc);
  } else {
    const int lg = R > 1 ? LOG : tbl_log2f_fast(h.deg, 4, 1, LOG);
    const unsigned size = 1u << lg;
    constexpr unsigned kNone = 0xffffu;
    unsigned claim[U];  // the slots this thread claimed: 16 bits a round
    bool ok = true;
#pragma unroll
    for (int u = 0; u < U; u++) claim[u] = 0xffffffffu;
#pragma unroll
    for (int x = 0; x < R; x++) {
      if (x > 0) {
        load_arcs(a, i, h.beg + x * (G * U), h.deg - x * (G * U), lane, G, U, r);
#pragma unroll
        for (int u = 0; u < U; u++) cc[u] = a.st.Cp[r.jj[u]];
      }
#pragma unroll
      for (int u = 0; u < U; u++) {
        if (r.jj[u] == i) continue;  // padding and i's self-loop
        if (cc[u] == d) {
          kid += r.ww[u];
        } else {
          bool own;
          const unsigned sl = tbl_put(tk, tv, size - 1, 32 - lg, cc[u], r.ww[u], &own);
          if (own) claim[u] = x ? ((claim[u] & 0xffffu) | (sl << 16)) : ((claim[u] & 0xffff0000u) | sl);
          ok &= sl < size;
        }
      }
    }
    if (!ok) atomicOr(&a.st.ctrl->error, kErrTableFull);
    A sg[U];
    if constexpr (R == 1) {  // the claimed communities' totals are on their way during the wait
#pragma unroll
      for (int u = 0; u < U; u++) sg[u] = (claim[u] & 0xffffu) != kNone ? sp.sr[cc[u]] : A(0);
    }
    if constexpr (G < 32) {
#pragma unroll
      for (int o = G / 2; o >= 1; o >>= 1) kid += __shfl_xor_sync(Grp<G>::mask(), kid, o);
    } else {
      __syncwarp();
      kid = warp_total(kid);
    }
    if (G > 32 && (lane & 31) == 0) sh.red_h[warp] = kid;
    team_sync<G, T>();  // every addition is made
    if constexpr (G > 32) kid = warp_total((threadIdx.x & 31) < G / 32 ? sh.red_h[gi * (G / 32) + (threadIdx.x & 31)] : H(0));
#pragma unroll
    for (int x = 0; x < R; x++) {
      int32_t key[U];
      H val[U];
#pragma unroll
      for (int u = 0; u < U; u++) {
        const unsigned sl = x ? claim[u] >> 16 : claim[u] & 0xffffu;
        key[u] = kEmpty;
        val[u] = H(0);
        if (sl != kNone) {
          key[u] = R > 1 ? tk[sl] : cc[u];
          val[u] = tv[sl];
          tk[sl] = kEmpty;
          tv[sl] = H(0);
        }
      }
      if constexpr (R > 1) {
#pragma unroll
        for (int u = 0; u < U; u++) sg[u] = key[u] != kEmpty ? sp.sr[key[u]] : A(0);
      }
#pragma unroll
      for (int u = 0; u < U; u++) {
        if (key[u] == kEmpty) continue;
        const S sc = sweep_score<M>(val[u], kid, ki, sg[u], sd, two_m);
        if (better(sc, key[u], best, bc)) { best = sc; bc = key[u]; }
      }
    }
    if constexpr (G < 32) {
      group_argmax<G>(best, bc);
    } else {
      __syncwarp();
      warp_best(best, bc);
    }
    if constexpr (G > 32) {
      if ((threadIdx.x & 31) == 0) {
        sh.red_s[warp] = best;
        sh.red_c[warp] = bc;
      }
      team_sync<G, T>();
      const bool in = (threadIdx.x & 31) < G / 32;
      best = in ? sh.red_s[gi * (G / 32) + (threadIdx.x & 31)] : M::lowest();
      bc = in ? sh.red_c[gi * (G / 32) + (threadIdx.x & 31)] : 0x7fffffff;
      warp_best(best, bc);
    } else {
      team_sync<G, T>();  // the table is empty again
    }
  }
  if (a.pruning && lane == 0) a.st.flags[i] = 0;
  if (bc != 0x7fffffff && best > S(0)) {
    if (lane == 0) sweep_move(a, sh, sp, i, d, bc, ki, best, gcv);
    if (a.pruning) {
      if constexpr (R > 1) {
        for (int e = lane; e < h.deg; e += G) {
          const int32_t j = a.g.tg[h.beg + e];
          if (j != i) a.st.flags[j] = 1;
        }
      } else {
#pragma unroll
        for (int u = 0; u < U; u++)
          if (r.jj[u] != i) a.st.flags[r.jj[u]] = 1;
      }
    }
  }
}

// The rows list[first], list[first + step], ... below cnt.  The first one's head h and, where flagged,
// arcs r are loaded; `sure`: h.on was read in this step.  (Loading the next row ahead here as well costs
// more registers than it hides: 5% slower throughout.)
template <class M, class R_, int T, int N>
__device__ __forceinline__ void sweep_rows(const SweepArgs<M>& a, SweepShared<M>& sh, const Step<M>& sp,
                                           const int32_t* list, unsigned first, unsigned cnt, unsigned step, Head<M>& h,
                                           Arcs<M, N>& r, bool sure) {
  constexpr int G = R_::G, U = R_::U;
  const int lane = threadIdx.x & (G - 1);
  bool loaded = h.on != 0;
  for (unsigned idx = first; idx < cnt; idx += step) {  // (counts are below 2^31)
    if (idx != first) {
      load_head(a, list[idx], h);
      sure = true;
      loaded = h.on != 0;
      if (loaded) load_arcs(a, h.i, h.beg, h.deg, lane, G, U, r);
    }
    sweep_row<M, R_, T>(a, sh, sp, h, r, loaded, sure);
  }
}

// ---------------------------------------------------------------- giants in the shared pool
// One warp reads the descriptors of giants [k, min(k + kSwPool, k1)) of the class list.
template <class M>
__device__ __forceinline__ void load_descs(const SweepArgs<M>& a, const int32_t* list, int64_t k, int64_t k1, GiantDesc* out) {
  const int lane = threadIdx.x & 31;
  if (k + lane >= k1) return;
  const GiantPlan& p = a.gp;
  GiantDesc g;
  g.k = k + lane;
  g.i = list[g.k];
  g.beg = a.g.rbeg[g.i];
  g.deg = (int)(a.g.rend[g.i] - g.beg);
  const int64_t t0 = p.tab_off[g.k];
  g.tab = t0 - p.tab_off[k];
  g.lg = 63 - __clzll(p.tab_off[g.k + 1] - t0);
  g.part = p.slice_off[g.k];
  g.pad = 0;
  out[lane] = g;
}

// Pieces of 32 * U arcs over the batch's giants: lane l holds giant l's end in the piece order.
template <int U>
__device__ __forceinline__ unsigned pool_pieces(const GiantDesc* gd, int ng, unsigned* total) {
  const int lane = threadIdx.x & 31;
  unsigned x = lane < ng ? ((unsigned)gd[lane].deg + 32 * U - 1) / (32 * U) : 0;  // at most 2^31 in all
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  *total = __shfl_sync(0xffffffffu, x, 31);
  return x;
}
// One arc a lane where the launch's pool blocks have a lane for every arc.
__device__ __forceinline__ bool pool_narrow(const GiantDesc* gd, int ng, unsigned blocks) {
  unsigned total;
  pool_pieces<1>(gd, ng, &total);
  return total <= blocks * kSwWarps;
}
// Giant and offset of piece t.
__device__ __forceinline__ int pool_find(unsigned end, unsigned t, unsigned* before) {
  const int k = __popc(__ballot_sync(0xffffffffu, end <= t));
  const unsigned e = __shfl_up_sync(0xffffffffu, end, 1);
  *before = __shfl_sync(0xffffffffu, (threadIdx.x & 31) == 0 ? 0 : e, k);
  return k;
}

template <class M, int U, int N>
__device__ __forceinline__ void pool_load(const SweepArgs<M>& a, const GiantDesc* gd, int ng, unsigned t, Head<M>& h,
                                          Arcs<M, N>& r) {
  unsigned total, before;
  const unsigned end = pool_pieces<U>(gd, ng, &total);
  h.i = -1;
  if (t >= total) return;
  const int k = pool_find(end, t, &before);
  h.i = gd[k].i;
  h.at = k;
  const int off = (int)(t - before) * (32 * U);
  load_arcs(a, h.i, gd[k].beg + off, min(gd[k].deg - off, 32 * U), threadIdx.x & 31, 32, U, r);
}

// Adds each lane's (key, w) (where `in`) to a pool table; all lanes of the warp call it.  A probe reads
// a bucket of four slots (one 32-byte sector).  The lanes go through a probe together -- one read, one
// compare-and-swap, both predicated -- since under a branch each would wait for its own atomic before
// the next lane's is issued (that way an insertion took 18,000 cycles, three waits take 4,000).  A
// claimed slot's bit is set in the pool's bitmap.
template <class V>
__device__ __forceinline__ bool pool_put(bool in, int32_t* kv, int lg, int32_t key, V w, unsigned* bits, int64_t base) {
  const unsigned mask = (1u << lg) - 1;
  const unsigned long long mine = ((unsigned long long)val_bits<V>(w) << 32) | (uint32_t)key;
  // the key's order of a bucket's slots starts at its home slot: fewer claims meet
  const unsigned home = tbl_home(key, 32 - lg), rot = home & 3u;
  unsigned s = home & ~3u;
  int32_t k[4] = {0, 0, 0, 0};
  bool left = in, load = in;
  unsigned from = 0;  // slots of the bucket, in that order, already found taken
  // a bucket takes at most five rounds: four claims lost to other keys, and one that finds none left
  const unsigned rounds = 5 * ((mask + 1) / 4);
  for (unsigned p = 0; __any_sync(0xffffffffu, left) && p < rounds; p++) {
    if (load) {
      const int4 x = __ldcg(reinterpret_cast<const int4*>(kv + 2 * (size_t)s));
      const int4 y = __ldcg(reinterpret_cast<const int4*>(kv + 2 * (size_t)s) + 1);
      const bool r1 = rot & 1u, r2 = rot & 2u;  // k[t] = key of slot (rot + t) & 3
      const int32_t b0 = r2 ? y.x : x.x, b1 = r2 ? y.z : x.z, b2 = r2 ? x.x : y.x, b3 = r2 ? x.z : y.z;
      k[0] = r1 ? b1 : b0; k[1] = r1 ? b2 : b1; k[2] = r1 ? b3 : b2; k[3] = r1 ? b0 : b3;
    }
    __syncwarp();
    // first slot that holds the key or is empty
    unsigned j = 4;
    bool hit = false;
#pragma unroll
    for (int t = 3; t >= 0; t--)
      if ((unsigned)t >= from && (k[t] == key || k[t] == kEmpty)) {
        j = t;
        hit = k[t] == key;
      }
    const bool claim = left && j < 4 && !hit;
    const unsigned at = s + ((rot + j) & 3u);
    unsigned long long old = 0;
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %1, 0;\n\tmov.b64 %0, 0;\n\t@q atom.global.cas.b64 %0, [%2], %3, %4;\n\t}"
                 : "=&l"(old)
                 : "r"((int)claim), "l"(kv + 2 * (size_t)at), "l"(kEmptyPair), "l"(mine)
                 : "memory");
    load = false;
    if (claim) {
      if (old == kEmptyPair) {
        atomicOr(&bits[(base + at) >> 5], 1u << ((base + at) & 31));
        left = false;
      } else if ((int32_t)(uint32_t)old == key) {
        hit = true;
      } else {
        from = j + 1;  // taken meanwhile by another key
      }
    }
    if (left && hit) {
      atomicAdd(slot_val<V>(kv, at), w);
      left = false;
    }
    if (left && j == 4) {
      s = (s + 4) & mask;
      from = 0;
      load = true;
    }
  }
  return !left;
}

// Arcs of the batch's flagged giants into their tables: pieces t, t + step, ...
template <class M, int U, int N>
__device__ __forceinline__ void pool_insert(const SweepArgs<M>& a, const GiantDesc* gd, int ng, unsigned act, int32_t dl,
                                            unsigned t, unsigned step, Head<M>& h, Arcs<M, N>& r, bool have) {
  typedef typename M::h_t H;
  const GiantPlan& p = a.gp;
  unsigned total;
  pool_pieces<U>(gd, ng, &total);
  bool ok = true;
  for (; t < total; t += step) {
    if (!have) pool_load<M, U>(a, gd, ng, t, h, r);
    have = false;
    const int k = h.at;
    const int32_t d = __shfl_sync(0xffffffffu, dl, k);
    if (!((act >> k) & 1u)) continue;
    int32_t cc[U];
#pragma unroll
    for (int u = 0; u < U; u++) cc[u] = a.st.Cp[r.jj[u]];
    H kid = H(0);
#pragma unroll
    for (int u = 0; u < U; u++) {
      const bool arc = r.jj[u] != h.i;  // neither padding nor a self-loop
      if (arc && cc[u] == d) kid += r.ww[u];
      ok &= pool_put(arc && cc[u] != d, p.slots + 2 * gd[k].tab, gd[k].lg, cc[u], r.ww[u], p.bits, gd[k].tab);
    }
    kid = warp_total(kid);
    if ((threadIdx.x & 31) == 0 && kid != H(0)) atomicAdd(reinterpret_cast<H*>(p.kid) + gd[k].k, kid);
  }
  if (!ok) atomicOr(&a.st.ctrl->error, kErrTableFull);
}

// Best candidate of every 1024-slot range of the flagged giants' tables: 128 threads a range, eight
// bitmap words a warp, a lane per slot of a word (coalesced).  Slots and bits are cleared.
template <class M>
__device__ __forceinline__ void pool_scan(const SweepArgs<M>& a, SweepShared<M>& sh, const Step<M>& sp,
                                          const GiantDesc* gd, int ng, unsigned act, int32_t dl) {
  typedef typename M::h_t H;
  typedef typename M::a_t A;
  typedef typename M::s_t S;
  constexpr int W = 8;
  const GiantPlan& p = a.gp;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, team = threadIdx.x >> 7;
  const bool mine = lane < ng && ((act >> lane) & 1u);
  // lane l: the end of giant l in the order of all ranges, and its state
  unsigned end = mine ? (gd[lane].lg > kRangeLog ? 1u << (gd[lane].lg - kRangeLog) : 1u) : 0;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, end, o);
    if (lane >= o) end += y;
  }
  const unsigned total = __shfl_sync(0xffffffffu, end, 31);
  if (team * gridDim.x + blockIdx.x >= total) return;  // (every warp of the launch reading these would queue)
  H kidl = H(0);
  A kil = A(0), sdl = A(0), tml = sh.two_m;
  if (mine) {
    const int32_t i = gd[lane].i;
    kidl = reinterpret_cast<const H*>(p.kid)[gd[lane].k];
    kil = a.st.K[i];
    sdl = sp.sr[dl];
    if (a.st.gc) {
      const GraphCtl& g = a.st.gc[a.st.vg[i]];
      tml = M::is_fp ? (A)g.two_m_f : (A)g.two_m_i;
    }
  }
  for (unsigned q = team * gridDim.x + blockIdx.x; q < total; q += gridDim.x * (kSwThreads / 128)) {
    unsigned before;
    const int k = pool_find(end, q, &before);
    const H kid = __shfl_sync(0xffffffffu, kidl, k);
    const A ki = __shfl_sync(0xffffffffu, kil, k), sd = __shfl_sync(0xffffffffu, sdl, k);
    const A two_m = __shfl_sync(0xffffffffu, tml, k);
    const int64_t sb = ((int64_t)(q - before) << kRangeLog) + (warp & 3) * (32 * W), ts = (int64_t)1 << gd[k].lg;
    int2* kv = reinterpret_cast<int2*>(p.slots) + gd[k].tab + sb;
    unsigned* wp = p.bits + ((gd[k].tab + sb) >> 5);
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
    team_sync<128, kSwThreads>();
    if ((threadIdx.x & 127) == 0) {
      for (int w = 1; w < 4; w++)
        if (better(sh.red_s[warp + w], sh.red_c[warp + w], best, bc)) { best = sh.red_s[warp + w]; bc = sh.red_c[warp + w]; }
      reinterpret_cast<S*>(p.part_s)[gd[k].part + (q - before)] = best;
      p.part_c[gd[k].part + (q - before)] = bc;
    }
    team_sync<128, kSwThreads>();
  }
}

// Moves the flagged giants whose best candidate gains and marks their neighbours: every warp that
// takes arcs of a giant reduces its ranges' candidates, the one with its first arcs moves it.
template <class M>
__device__ __forceinline__ void pool_decide(const SweepArgs<M>& a, SweepShared<M>& sh, const Step<M>& sp,
                                            const GiantDesc* gd, int ng, unsigned act, int32_t dl) {
  typedef typename M::s_t S;
  constexpr int U = 4;
  const GiantPlan& p = a.gp;
  const int lane = threadIdx.x & 31;
  unsigned total;
  const unsigned end = pool_pieces<U>(gd, ng, &total);
  for (unsigned t = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; t < total; t += gridDim.x * kSwWarps) {
    unsigned before;
    const int k = pool_find(end, t, &before);
    const int32_t d = __shfl_sync(0xffffffffu, dl, k);
    if (!((act >> k) & 1u)) continue;
    const int32_t i = gd[k].i;
    const int off = (int)(t - before) * (32 * U);
    int32_t jj[U];
#pragma unroll
    for (int u = 0; u < U; u++) jj[u] = a.pruning && off + lane + u * 32 < gd[k].deg ? a.g.tg[gd[k].beg + off + lane + u * 32] : i;
    S best = M::lowest();
    int32_t bc = 0x7fffffff;
    const int64_t x1 = gd[k].part + (gd[k].lg > kRangeLog ? 1 << (gd[k].lg - kRangeLog) : 1);
    for (int64_t x = gd[k].part + lane; x < x1; x += 32) {
      const S s = reinterpret_cast<const S*>(p.part_s)[x];
      const int32_t c = p.part_c[x];
      if (better(s, c, best, bc)) { best = s; bc = c; }
    }
    __syncwarp();
    warp_best(best, bc);
    const bool mv = bc != 0x7fffffff && best > S(0);
    if (off == 0 && lane == 0) {
      reinterpret_cast<uint32_t*>(p.kid)[gd[k].k] = 0u;  // for the next use of the plan (0u is also 0.0f)
      if (a.pruning) a.st.flags[i] = 0;
      if (mv) sweep_move(a, sh, sp, i, d, bc, a.st.K[i], best, a.st.gc ? a.st.gc + a.st.vg[i] : nullptr);
    }
    if (mv) {
#pragma unroll
      for (int u = 0; u < U; u++)
        if (jj[u] != i) a.st.flags[jj[u]] = 1;
    }
  }
}

// ---------------------------------------------------------------- blocks by kind of row
// With several blocks every block takes one kind of row, so that the kinds run side by side and each
// group's first row can be loaded a step ahead: kind x has the blocks up to byte x of the record's word
// (0: rows of a block with 4097-8192 arcs, 1-6: degree buckets 5-0), the pool giants the blocks after
// those.
__device__ __forceinline__ int role_end(unsigned long long roles, int x) { return (int)((roles >> (8 * x)) & 255u); }
// First row of group gi (of `groups` a block) of a kind that has `nb` blocks, this one the b-th: few rows
// spread over the blocks, many run along neighbouring groups, which read neighbouring vertices' state.
__device__ __forceinline__ unsigned role_first(unsigned gi, unsigned groups, unsigned b, unsigned nb, unsigned cnt) {
  return cnt > nb * groups ? b * groups + gi : gi * nb + b;
}
__device__ __forceinline__ int role_of(unsigned long long roles, int block) {
  int x = 0;
  while (x < 7 && block >= role_end(roles, x)) x++;
  return x;
}

// Algorithm 2's tolerance test: 2 sum N <= tau (2m)^2 (the arithmetic of lm_finish).
template <bool FP>
__device__ __forceinline__ bool sweep_converged(unsigned long long lo, unsigned long long hi, double f, double tau,
                                                long long two_m_i, double two_m_f) {
  if (FP) return __dmul_rn(2.0, f) <= __dmul_rn(tau, __dmul_rn(two_m_f, two_m_f));
  const double t = __ll2double_rn(two_m_i);
  return u128_to_double_rn((hi << 1) | (lo >> 63), lo << 1) <= __dmul_rn(tau, __dmul_rn(t, t));
}

// Threads and arcs a thread of a kind of row.
template <int G_, int U_, int LOG_, int R_ = 1>
struct Role {
  static constexpr int G = G_, U = U_, LOG = LOG_, R = R_;
};

template <class M, int SC, bool HUBS>
__global__ void __launch_bounds__(HUBS ? kSwThreads : kSwLowThreads, 1) lm_sweep(SweepArgs<M> a, PersistBar bar) {
  typedef typename M::a_t A;
  typedef typename M::h_t H;
  constexpr int T = HUBS ? kSwThreads : kSwLowThreads, W = T / 32;
  extern __shared__ __align__(16) unsigned char sw_dyn[];
  SweepShared<M>& sh = *reinterpret_cast<SweepShared<M>*>(sw_dyn);
  Ctrl* const ctrl = a.st.ctrl;
  if (*(volatile int32_t*)&ctrl->done) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int t = tid; t < kSwSlots; t += T) { sh.keys[t] = kEmpty; sh.vals[t] = H(0); }
  if (tid < 2 * kStepWords) sh.rec[tid / kStepWords][tid % kStepWords] = a.recs[(tid / kStepWords) % a.nsteps * kStepWords + tid % kStepWords];
  if (tid < 3) sh.n_moves[tid] = 0;
  if (tid == 0) { sh.lo = sh.hi = sh.mv = 0; sh.f = 0.0; sh.done = 0; }
  for (int64_t c = (int64_t)blockIdx.x * T + tid; c < a.n_sig; c += (int64_t)gridDim.x * T)
    a.sig2[c] = a.st.Sig[c];
  __syncthreads();
  if (HUBS && warp == 0) load_descs(a, a.glist + sh.rec[0][kStepGiant], sh.rec[0][kStepLong], sh.rec[0][kStepGiant + 2], sh.gd[0]);
  if (tid == 0) sh.two_m = M::is_fp ? (A)ctrl->two_m_f : (A)ctrl->two_m_i;
  Head<M> head;
  Arcs<M, HUBS ? 8 : 4> arcs;
  // between the arrival at step n's barrier and the wait: the record of step n + 3, the pool giants of
  // step n + 2, and this thread's row of step n + 1
  auto ahead = [&](int n, int s) {
    if (warp == W - 1) {
      if (lane < kStepWords) sh.rec[(n + 3) & 3][lane] = a.recs[(int64_t)((s + 3) % a.nsteps) * kStepWords + lane];
    } else if (HUBS && warp == W - 2) {
      const int64_t* r2 = sh.rec[(n + 2) & 3];
      load_descs(a, a.glist + r2[kStepGiant], r2[kStepLong], r2[kStepGiant + 2], sh.gd[(n + 2) % 3]);
    }
    const int64_t* r = sh.rec[(n + 1) & 3];
    const unsigned long long roles = a.all_wide ? 0 : (unsigned long long)r[kStepRoles];
    head.i = -1;
    if (roles == 0) return;
    const int x = role_of(roles, blockIdx.x), b0 = x ? role_end(roles, x - 1) : 0;
    if (x < 7) {
      // log2 of the group size and arcs a thread: 512 512 256 64 32 8 4 threads, 8 8 8 8 4 2 1 arcs;
      // without hubs - - - 128 32 8 4 threads, 4 4 2 1 arcs
      const int lg = (int)(((HUBS ? 0x2356899u : 0x2357000u) >> (4 * x)) & 15u);
      const int U = (int)(((HUBS ? 0x1248888u : 0x1244000u) >> (4 * x)) & 15u);
      const int bk = 2 * (6 - x);
      const unsigned cnt = (unsigned)(x ? r[bk + 1] : r[kStepLong] - r[kStepGiant + 1]);
      const unsigned idx = role_first(tid >> lg, T >> lg, blockIdx.x - b0, role_end(roles, x) - b0, cnt);
      if (idx < cnt) {
        load_head(a, x ? a.perm[r[bk] + idx] : a.glist[r[kStepGiant] + r[kStepGiant + 1] + idx], head);
        if (head.on) load_arcs(a, head.i, head.beg, head.deg, tid & ((1 << lg) - 1), 1 << lg, U, arcs);
      }
    } else if constexpr (HUBS) {
      const int ng = (int)min((int64_t)kSwPool, r[kStepGiant + 2] - r[kStepLong]);
      const unsigned blocks = gridDim.x - b0, t = warp * blocks + (blockIdx.x - b0);
      const GiantDesc* gd = sh.gd[(n + 1) % 3];
      if (ng > 0) {
        if (pool_narrow(gd, ng, blocks)) pool_load<M, 1>(a, gd, ng, t, head, arcs);
        else pool_load<M, 4>(a, gd, ng, t, head, arcs);
      }
    }
  };
  unsigned long long sum;
  auto none = []() { return 0ULL; };
  int par = 0;           // Sigma copy that the step reads
  int n = -1, s = -1;    // step of the launch and of the iteration: the moves of step n are in list n % 2,
                         // their number in n_moves[n % 3]
  int it = 0;            // iterations finished
  while (true) {
    // end of step n (the start, n = -1, too)
    const bool ok = scope_barrier<SC>(
        bar, ctrl, &sum,
        [&]() {  // thread 0: the block's sums of the iteration travel with its last step's barrier
          if (s + 1 == a.nsteps && a.whole && !a.st.gc) {
            unsigned long long* t = a.state + kSwSums + 4 * (it % 3);
            if (sh.mv) {
              atomicAdd(&t[3], sh.mv);
              if (M::is_fp) atomicAdd(reinterpret_cast<double*>(&t[2]), sh.f);
              else atomic_add_u128(&t[0], &t[1], sh.lo, sh.hi);
            }
            sh.lo = sh.hi = sh.mv = 0;
            sh.f = 0.0;
          }
          return 0ULL;
        },
        [&]() { ahead(n, s); });
    if (!ok) return;
    if (n >= 0) {
      const int64_t* rec = sh.rec[n & 3];
      if (a.all_wide || rec[kStepWide]) {
        const int64_t v0 = rec[kStepApply], v1 = v0 + rec[kStepApply + 1];
        for (int64_t v = v0 + (int64_t)blockIdx.x * T + tid; v < v1; v += (int64_t)gridDim.x * T) {
          const int32_t i = a.perm[v], to = a.st.mv_to[i];
          if (to < 0) continue;
          const int32_t from = a.st.mv_from[i];
          const A ki = a.st.K[i];
          atomic_add_a(&a.st.Sig[from], -ki);
          atomic_add_a(&a.st.Sig[to], ki);
          atomic_add_a(&a.sig2[from], -ki);
          atomic_add_a(&a.sig2[to], ki);
          a.st.mv_to[i] = -1;
        }
        if (!scope_barrier<SC>(bar, ctrl, &sum, none)) return;
      }
      par ^= 1;
      if (tid == 0) sh.n_moves[(n + 2) % 3] = 0;  // read in this step, filled in the step after next
    }
    n++;
    if (++s == a.nsteps) {
      s = 0;
      if (!a.whole) break;
      it++;
      bool stop;
      if (a.st.gc) {
        // per graph; the graphs left come with the barrier
        const double tau = ctrl->tau;
        int left = 0;
        for (int g = blockIdx.x * T + tid; g < a.n_graphs; g += gridDim.x * T) {
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
    {
      const int64_t* rec = sh.rec[n & 3];
      Step<M> sp;
      sp.sr = par ? a.sig2 : a.st.Sig;
      sp.sw = par ? a.st.Sig : a.sig2;
      sp.wide = a.all_wide || rec[kStepWide] != 0;
      sp.nb = n & 1;
      sp.n_moves = &sh.n_moves[n % 3];
      const unsigned long long roles = a.all_wide ? 0 : (unsigned long long)rec[kStepRoles];
      // the last step's moves on the copy that lacks them
      {
        const SweepMove<M>* mv = sh.moves[(n + 1) & 1];
        const int nm = min(sh.n_moves[(n + 2) % 3], kSwMoves);
        for (int t = tid; t < nm; t += T) {
          atomic_add_a(&sp.sw[mv[t].from], -mv[t].k);
          atomic_add_a(&sp.sw[mv[t].to], mv[t].k);
        }
      }
      // pool giants (a batch of at most 32): lane l holds giant l's community, act the flagged ones
      const GiantDesc* gd = sh.gd[n % 3];
      int ng = (int)min((int64_t)kSwPool, rec[kStepGiant + 2] - rec[kStepLong]);
      unsigned act = 0;
      int32_t dl = 0;
      [[maybe_unused]] auto activate = [&]() {
        bool on = false;
        if (lane < ng) {
          const int32_t i = gd[lane].i;
          dl = a.st.Cp[i];
          on = (!a.pruning || a.st.flags[i] != 0) && !(a.st.gc && *(volatile int32_t*)&a.st.gc[a.st.vg[i]].done);
        }
        act = __ballot_sync(0xffffffffu, on);
      };
      [[maybe_unused]] auto insert = [&](int b0, bool have) {
        const unsigned blocks = gridDim.x - b0;
        if ((int)blockIdx.x < b0) return;
        const unsigned t = warp * blocks + (blockIdx.x - b0);
        if (pool_narrow(gd, ng, blocks)) pool_insert<M, 1>(a, gd, ng, act, dl, t, blocks * W, head, arcs, have);
        else pool_insert<M, 4>(a, gd, ng, act, dl, t, blocks * W, head, arcs, have);
      };
      if constexpr (HUBS) if (ng > 0) {
        activate();
        insert(roles ? role_end(roles, 6) : 0, roles && head.i >= 0);
      }
      // rows: one kind a block, or (one block) every kind, long rows first
      auto rows = [&](auto tag, int x, const int32_t* rl, unsigned cnt) {
        constexpr int G = decltype(tag)::G, U = decltype(tag)::U, GPB = T / G;
        if (cnt == 0) return;
        const int gi = tid / G;
        unsigned first, step = gridDim.x * GPB;
        if (roles) {
          const int b0 = x ? role_end(roles, x - 1) : 0, b1 = role_end(roles, x);
          if ((int)blockIdx.x < b0 || (int)blockIdx.x >= b1) return;
          first = role_first(gi, GPB, blockIdx.x - b0, b1 - b0, cnt);
          step = (b1 - b0) * GPB;
        } else {
          first = role_first(gi, GPB, blockIdx.x, gridDim.x, cnt);
        }
        if (!roles && first < cnt) {
          load_head(a, rl[first], head);
          if (head.on) load_arcs(a, head.i, head.beg, head.deg, tid & (G - 1), G, U, arcs);
        }
        sweep_rows<M, decltype(tag), T>(a, sh, sp, rl, first, cnt, step, head, arcs, roles == 0);
        // Where one block takes every kind, the next kind's smaller groups write red_s and red_c: not
        // before every warp of this group has read its last row's candidates there.
        if constexpr (HUBS && G > 32)
          if (!roles) team_sync<G, T>();
      };
      if constexpr (HUBS) {
        rows(Role<512, 8, 14, 2>(), 0, a.glist + rec[kStepGiant] + rec[kStepGiant + 1],
             (unsigned)(rec[kStepLong] - rec[kStepGiant + 1]));
        rows(Role<512, 8, 14>(), 1, a.perm + rec[10], (unsigned)rec[11]);
        rows(Role<256, 8, 13>(), 2, a.perm + rec[8], (unsigned)rec[9]);
        rows(Role<64, 8, 11>(), 3, a.perm + rec[6], (unsigned)rec[7]);
      } else {
        rows(Role<128, 4, 11>(), 3, a.perm + rec[6], (unsigned)rec[7]);
      }
      rows(Role<32, 4, 9>(), 4, a.perm + rec[4], (unsigned)rec[5]);
      rows(Role<8, 2, 6>(), 5, a.perm + rec[2], (unsigned)rec[3]);
      rows(Role<4, 1, 3>(), 6, a.perm + rec[0], (unsigned)rec[1]);
      if constexpr (HUBS) if (ng > 0) {
        for (int64_t kb = rec[kStepLong];;) {
          if (!scope_barrier<SC>(bar, ctrl, &sum, [&]() { return act ? 1ULL : 0ULL; })) return;
          if (sum & kBarSum) {  // some giant of the batch is flagged
            pool_scan<M>(a, sh, sp, gd, ng, act, dl);
            if (!scope_barrier<SC>(bar, ctrl, &sum, none)) return;
            pool_decide<M>(a, sh, sp, gd, ng, act, dl);
          }
          kb += kSwPool;
          if (kb >= rec[kStepGiant + 2]) break;
          __syncthreads();
          if (HUBS && warp == 0) load_descs(a, a.glist + rec[kStepGiant], kb, rec[kStepGiant + 2], sh.gdx);
          // the tables of the last batch are empty once every block has scanned them
          if (!scope_barrier<SC>(bar, ctrl, &sum, none)) return;
          gd = sh.gdx;
          ng = (int)min((int64_t)kSwPool, rec[kStepGiant + 2] - kb);
          activate();
          insert(0, false);
        }
      }
    }
  }
  // both copies hold every move in the end
  {
    const SweepMove<M>* mv = sh.moves[(n + 1) & 1];
    const int nm = min(sh.n_moves[(n + 2) % 3], kSwMoves);
    A* const s = par ? a.st.Sig : a.sig2;
    for (int t = tid; t < nm; t += T) {
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

// The giants of every step's perm range, class after class (records hold both places).
__global__ void k_collect_giants(const int64_t* recs, int nsteps, const int32_t* perm, int32_t* glist) {
  for (int s = blockIdx.x * (kBlock / 32) + threadIdx.x / 32; s < nsteps; s += gridDim.x * (kBlock / 32)) {
    const int64_t* r = recs + (int64_t)s * kStepWords;
    const int64_t k0 = r[kStepGiant + 1], cnt = r[kStepGiant + 2] - k0;
    const int64_t from = r[kStepApply] + r[kStepApply + 1] - cnt;  // a class's last rows
    for (int64_t t = threadIdx.x & 31; t < cnt; t += 32) glist[k0 + t] = perm[from + t];
  }
}
void collect_giants(Ctx& c, const int64_t* recs, int nsteps, const int32_t* perm, int32_t* glist) {
  k_collect_giants<<<grid_for(nsteps, kBlock / 32, c.num_sms), kBlock, 0, c.s>>>(recs, nsteps, perm, glist);
  c.launches++;
}

template <class M, bool HUBS>
static cudaError_t sweep_launch(Scope sc, const Ctx& c, const SweepArgs<M>& a, const PersistBar& bar) {
  constexpr size_t smem = sizeof(SweepShared<M>);
  constexpr int T = HUBS ? kSwThreads : kSwLowThreads;
  if (sc == kCta) return scope_launch(sc, c, lm_sweep<M, kCta, HUBS>, T, smem, a, bar);
  if (sc == kCluster) return scope_launch(sc, c, lm_sweep<M, kCluster, HUBS>, T, smem, a, bar);
  return scope_launch(sc, c, lm_sweep<M, kGrid, HUBS>, T, smem, a, bar);
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
  const long long spins = c.step_spins > 0 ? c.step_spins : c.wait_spins;
  const PersistBar bar{sw.state + kSwBar, spins > 0 ? spins : kBarrierPolls, 0, c.step_from};
  // a caller that bounds the waits gets the bounded barrier
  const Scope sc = spins > 0 ? kGrid : (Scope)sw.scope;
  e = sw.hubs ? sweep_launch<M, true>(sc, c, a, bar) : sweep_launch<M, false>(sc, c, a, bar);
  if (e != cudaSuccess && sc != kCta) {  // the scope cannot be launched here: one block can
    cudaGetLastError();
    a.all_wide = 1;
    e = sw.hubs ? sweep_launch<M, true>(kCta, c, a, bar) : sweep_launch<M, false>(kCta, c, a, bar);
  }
  c.launches++;
  return e;
}

template cudaError_t move_sweep<IntMode>(Ctx&, const SweepPlan&, const GraphView<int32_t>&, const PassState<IntMode>&,
                                         const int32_t*, const int32_t*, const GiantPlan&, bool, int32_t);
template cudaError_t move_sweep<FpMode>(Ctx&, const SweepPlan&, const GraphView<float>&, const PassState<FpMode>&,
                                        const int32_t*, const int32_t*, const GiantPlan&, bool, int32_t);

}  // namespace lv
