// move.cu -- the local-moving phase of Algorithm 2 on the GPU.
//
// One group of G threads handles one vertex i (G by degree bucket: 4, 8, 32 lanes or a block of
// 128 or 512 threads; rows above 4096 arcs take the multi-block path of giant.cu, whose tables live in global
// memory).  The group takes i's arcs (scanCommunities with self = false), accumulates
// K_i->c for every neighbouring community c != C'[i] in an open-addressing table in shared
// memory and K_i->d in registers, then scores
// every candidate with the Eq. 2 numerator
//     N(c) = 2m (K_i->c - K_i->d) - K_i (Sigma_c - Sigma_d + K_i)
// (exact int64 for int32 weights), takes the best with ties to the smallest id and moves iff
// N > 0.  Deterministic mode records the move and defers the Sigma update to move_apply (the
// colour class decides against class-start totals); fast mode applies it at once with atomics.
// A moved vertex re-marks its neighbours for processing (vertex pruning, Section 4.1.6).  The
// sum of the performed N is accumulated exactly (128-bit) and move_finish applies the
// per-iteration tolerance test of Algorithm 2 on the device, so iterations need no host sync.
#include <atomic>
#include <type_traits>

#include "internal.cuh"

namespace lv {

template <class M>
struct LmArgs {
  GraphView<typename M::w_t> g;
  PassState<M> st;
  const int32_t* list;
  int64_t count;
  int fast;
  int pruning;
  int bucket;
  const int64_t* rng;  // device {start, count} of the list (a captured iteration), or null
  int tf;              // table slots per key of the row's distinct-key bound
};

// Block-wide reduction of the per-thread move accumulators into the control block.
template <bool FP>
__device__ __forceinline__ void flush_move_acc(Ctrl* ctrl, unsigned long long lo, unsigned long long hi,
                                               unsigned long long mv, double f, unsigned long long* s_lo,
                                               unsigned long long* s_hi, unsigned long long* s_mv, double* s_f) {
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    unsigned long long lo2 = __shfl_xor_sync(0xffffffffu, lo, o);
    unsigned long long hi2 = __shfl_xor_sync(0xffffffffu, hi, o);
    unsigned long long s = lo + lo2;
    hi += hi2 + (s < lo ? 1ULL : 0ULL);
    lo = s;
    mv += __shfl_xor_sync(0xffffffffu, mv, o);
    if (FP) f += __shfl_xor_sync(0xffffffffu, f, o);
  }
  __syncthreads();
  if ((threadIdx.x & 31) == 0) {
    s_lo[threadIdx.x >> 5] = lo; s_hi[threadIdx.x >> 5] = hi; s_mv[threadIdx.x >> 5] = mv; s_f[threadIdx.x >> 5] = f;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long tl = 0, th = 0, tm = 0;
    double tf = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) {
      unsigned long long s = tl + s_lo[w];
      th += s_hi[w] + (s < tl ? 1ULL : 0ULL);
      tl = s;
      tm += s_mv[w];
      tf += s_f[w];
    }
    if (tm) {
      atomicAdd(&ctrl->moves, tm);
      if (FP) atomicAdd(&ctrl->sum_f, tf);
      else atomic_add_u128(&ctrl->sum_lo, &ctrl->sum_hi, tl, th);
    }
  }
}

// Shape of a bucket's kernel: G threads a row, U arcs a thread, R rounds of them (G * U * R arcs hold the
// bucket's longest row), tables of 2^LOG slots, blocks of T threads, B of them an SM (64 registers a
// thread, 32 warps an SM).
template <int G_, int U_, int R_, int LOG_, int T_, int B_>
struct LmShape {
  static constexpr int G = G_, U = U_, R = R_, LOG = LOG_, T = T_, B = B_, GPB = T_ / G_;
  static constexpr bool kTable = G > 4;
  template <class H>
  static constexpr size_t smem() { return kTable ? (size_t)GPB * (1 << LOG) * (sizeof(int32_t) + sizeof(H)) : 0; }
};
typedef LmShape<4, 1, 1, 0, 256, 4> Lm0;
typedef LmShape<8, 2, 1, 6, 256, 4> Lm1;
typedef LmShape<32, 4, 1, 9, 128, 8> Lm2;
typedef LmShape<128, 4, 1, 11, 128, 8> Lm3;
typedef LmShape<512, 4, 1, 13, 512, 2> Lm4;
typedef LmShape<512, 4, 2, 13, 512, 2> Lm5;

// One group per row.  Bound by the chain of dependent loads of a row and by how many rows an SM holds, so:
// a row fits its group in one step (its targets stay in registers for the marks); the next row's head is
// loaded during this one; the U swaps of a thread go out together; the thread that claims a slot loads
// that community's Sigma at once and scores and clears the slot, without a list of claims; tables are a
// quarter full where shared memory allows (half full, a 4096-arc row probes 2.5 times as long).
// R-MAT 22 fast, ms of a run in rows of 129-512 arcs 4.88 -> 3.65, 513-2048 3.75 -> 3.43, 2049-4096
// 3.49 -> 2.46, 17-128 3.23 -> 2.90, 5-16 1.27 -> 1.03, 1-4 0.94 -> 0.80, against a warp for up to 512 arcs
// and 256 threads beyond, in rounds of four arcs a thread (the run 28.9 -> 23.8).  L1 and L2 then move
// half of what they could and 37% of the issue slots are used: the rest is latency at 30 warps an SM.
// Other shapes: 64 threads of eight arcs for 129-512 4.45, 256 of eight for 513-2048 3.71, 1024 of four
// for 2049-4096 2.75 (and it holds the whole SM), 16 lanes of eight for 17-128 4.32, 24 warps of 85
// registers even.
template <class M, class P>
__global__ void __launch_bounds__(P::T, P::B) lm_kernel(LmArgs<M> a) {
  typedef typename M::h_t H;
  typedef typename M::a_t A;
  typedef typename M::s_t S;
  constexpr int G = P::G, U = P::U, R = P::R, LOG = P::LOG, T = P::T, GPB = P::GPB, NW = T / 32;
  static_assert(G <= 32 || G == T, "a group is lanes of a warp or the block");
  Ctrl* ctrl = a.st.ctrl;
  if (*(volatile int32_t*)&ctrl->done) return;
  // a captured iteration reads its list range from device memory (32-bit: counts and offsets are
  // below 2^31); the graph's arrays stay kernel parameters
  unsigned lo = 0, hi = (unsigned)a.count;  // list[lo, hi)
  if (a.rng) {
    lo = (unsigned)a.rng[0];
    hi = lo + (unsigned)a.rng[1];
  }
  if (lo + blockIdx.x * GPB >= hi) return;  // a fixed grid larger than this range
  const GraphView<typename M::w_t>& g = a.g;
  extern __shared__ __align__(16) unsigned char lm_dyn[];  // GPB tables of 2^LOG (key, value) slots
  const int gi = threadIdx.x / G, lane = threadIdx.x & (G - 1);
  int32_t* const tk = reinterpret_cast<int32_t*>(lm_dyn) + (gi << LOG);
  H* const tv = reinterpret_cast<H*>(lm_dyn + sizeof(int32_t) * (GPB << LOG)) + (gi << LOG);
  __shared__ S red_s[NW];
  __shared__ int32_t red_c[NW];
  __shared__ H red_h[NW];
  __shared__ int32_t red_i[1];
  __shared__ unsigned long long r_lo[NW], r_hi[NW], r_mv[NW];
  __shared__ double r_f[NW];
  if constexpr (P::kTable) {
    // 16 bytes a store; value 0 is 0u and 0.0f
    for (int t = lane; t < (1 << LOG) / 4; t += G) {
      reinterpret_cast<int4*>(tk)[t] = make_int4(kEmpty, kEmpty, kEmpty, kEmpty);
      reinterpret_cast<int4*>(tv)[t] = make_int4(0, 0, 0, 0);
    }
    Grp<G>::sync();
  }
  const A two_m_all = M::is_fp ? (A)ctrl->two_m_f : (A)ctrl->two_m_i;
  GraphCtl* const gcs = a.st.gc;
  unsigned long long acc_lo = 0, acc_hi = 0, arcs = 0;
  double acc_f = 0.0;
  unsigned listed = 0, processed = 0, cand = 0, moved = 0, marks = 0;

  const unsigned stride = gridDim.x * GPB;
  unsigned idx = lo + blockIdx.x * GPB + gi;
  int32_t i1 = 0, i2 = 0, vg1 = 0;  // the next row, its head, and the one after it
  int64_t b1 = 0, e1 = 0;
  A k1 = A(0);
  if (idx < hi) {
    i1 = a.list[idx];
    b1 = g.rbeg[i1];
    e1 = g.rend[i1];
    k1 = a.st.K[i1];
    if (gcs) vg1 = a.st.vg[i1];
    if (hi - idx > stride) i2 = a.list[idx + stride];
  }
  for (bool more = idx < hi; more;) {
    const int32_t i = i1;
    const int64_t beg = b1;
    const int deg = (int)(e1 - b1);
    const A ki = k1;
    GraphCtl* const gcv = gcs ? gcs + vg1 : nullptr;  // batched run: the graph of i
    const int32_t d = a.st.Cp[i];
    // every thread reads the flag and the group takes the OR, so the decision is uniform even if a
    // neighbour re-marks i meanwhile; then i is marked as processed
    bool on = !a.pruning || a.st.flags[i] != 0;
    A two_m = two_m_all;
    if (gcv) {
      on = on && !*(volatile int32_t*)&gcv->done;  // skipped once its local-moving phase has converged
      two_m = M::is_fp ? (A)gcv->two_m_f : (A)gcv->two_m_i;
    }
    more = hi - idx > stride;
    idx += stride;
    if (more) {
      i1 = i2;
      b1 = g.rbeg[i1];
      e1 = g.rend[i1];
      k1 = a.st.K[i1];
      if (gcs) vg1 = a.st.vg[i1];
      if (hi - idx > stride) i2 = a.list[idx + stride];
    }
    if (lane == 0) listed++;
    if (!group_any<G>(on)) continue;
    if (lane == 0) {
      if (a.pruning) a.st.flags[i] = 0;
      processed++;
      arcs += (unsigned long long)deg;
    }
    const int32_t* const rtg = g.tg + beg;
    const typename M::w_t* const rw = g.w + beg;
    int32_t jj[U], cc[U];
    H ww[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
      const int e = lane + u * G;
      jj[u] = e < deg ? rtg[e] : i;
      ww[u] = e < deg ? (H)rw[e] : H(0);
    }
    const A sd = a.st.Sig[d];
    const int32_t lone = a.fast && lane == 0 ? a.st.csize[d] : 0;
#pragma unroll
    for (int u = 0; u < U; u++) cc[u] = a.st.Cp[jj[u]];

    H kid = H(0);
    S best = M::lowest();
    int32_t bc = 0x7fffffff;
    if constexpr (!P::kTable) {  // four arcs: the lanes compare their communities
      const unsigned m = Grp<G>::mask();
      const bool self = jj[0] == i;  // padding and i's self-loop
      if (self) cc[0] = d;
      H same = ww[0];
      bool lower = false;
#pragma unroll
      for (int o = 1; o < G; o++) {
        const int32_t c2 = __shfl_xor_sync(m, cc[0], o);
        const H w2 = __shfl_xor_sync(m, ww[0], o);
        if (c2 == cc[0]) {
          same += w2;
          lower |= (lane ^ o) < lane;
        }
      }
      const bool own = cc[0] != d && !lower;
      const A sg = own ? a.st.Sig[cc[0]] : A(0);
      kid = group_sum<G>(!self && cc[0] == d ? ww[0] : H(0), (H*)nullptr);
      if (own) {
        cand++;
        best = M::score(same, kid, ki, sg, sd, two_m);
        bc = cc[0];
      }
      group_argmax<G>(best, bc);
    } else {
      const int lg = tbl_log2f_fast(deg, 2 * a.tf, 1, LOG);
      const unsigned mask = (1u << lg) - 1;
      unsigned claim[U];  // the slots this thread claimed: 16 bits a round
      bool ok = true;
#pragma unroll
      for (int u = 0; u < U; u++) claim[u] = 0xffffffffu;
#pragma unroll
      for (int x = 0; x < R; x++) {
        if (x > 0) {
#pragma unroll
          for (int u = 0; u < U; u++) {
            const int e = lane + (x * U + u) * G;
            jj[u] = e < deg ? rtg[e] : i;
            ww[u] = e < deg ? (H)rw[e] : H(0);
          }
#pragma unroll
          for (int u = 0; u < U; u++) cc[u] = a.st.Cp[jj[u]];
        }
        unsigned s[U];
        bool in[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
          in[u] = jj[u] != i && cc[u] != d;
          if (jj[u] != i && cc[u] == d) kid += ww[u];
        }
        const unsigned own = tbl_put<U>(in, tk, tv, mask, 32 - lg, cc, ww, s, &ok);
#pragma unroll
        for (int u = 0; u < U; u++)
          if ((own >> u) & 1u) claim[u] = x ? ((claim[u] & 0xffffu) | (s[u] << 16)) : ((claim[u] & 0xffff0000u) | s[u]);
      }
      if (!ok) atomicOr(&ctrl->error, kErrTableFull);
      A sg[U];
      if constexpr (R == 1) {  // the claimed communities' totals are on their way during the wait
#pragma unroll
        for (int u = 0; u < U; u++) sg[u] = (claim[u] & 0xffffu) != 0xffffu ? a.st.Sig[cc[u]] : A(0);
      }
      if constexpr (G < 32) {
        kid = group_sum<G>(kid, (H*)nullptr);
      } else {
        __syncwarp();
        kid = warp_total(kid);
      }
      if (G > 32 && (threadIdx.x & 31) == 0) red_h[threadIdx.x >> 5] = kid;
      Grp<G>::sync();  // every addition is made
      if constexpr (G > 32) kid = warp_total((threadIdx.x & 31) < NW ? red_h[threadIdx.x & 31] : H(0));
#pragma unroll
      for (int x = 0; x < R; x++) {
        int32_t key[U];
        H val[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
          const unsigned sl = x ? claim[u] >> 16 : claim[u] & 0xffffu;
          key[u] = kEmpty;
          val[u] = H(0);
          if (sl != 0xffffu) {
            key[u] = R > 1 ? tk[sl] : cc[u];
            val[u] = tv[sl];
            tk[sl] = kEmpty;
            tv[sl] = H(0);
          }
        }
        if constexpr (R > 1) {
#pragma unroll
          for (int u = 0; u < U; u++) sg[u] = key[u] != kEmpty ? a.st.Sig[key[u]] : A(0);
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
          if (key[u] == kEmpty) continue;
          cand++;
          const S sc = M::score(val[u], kid, ki, sg[u], sd, two_m);
          if (better(sc, key[u], best, bc)) { best = sc; bc = key[u]; }
        }
      }
      if constexpr (G < 32) {
        group_argmax<G>(best, bc);
        Grp<G>::sync();  // the table is empty again
      } else {
        __syncwarp();  // for a warp's row: the table is empty again
        warp_best(best, bc);
      }
      if constexpr (G > 32) {
        if ((threadIdx.x & 31) == 0) {
          red_s[threadIdx.x >> 5] = best;
          red_c[threadIdx.x >> 5] = bc;
        }
        __syncthreads();
        const bool in = (threadIdx.x & 31) < NW;
        best = in ? red_s[threadIdx.x & 31] : M::lowest();
        bc = in ? red_c[threadIdx.x & 31] : 0x7fffffff;
        warp_best(best, bc);
      }
    }

    int mv = (bc != 0x7fffffff && best > S(0)) ? 1 : 0;
    if (mv && a.fast) {
      // singleton guard against lock-step swaps: a lone vertex joins another singleton
      // community only if that community's id is smaller
      int okm = 1;
      if (lane == 0 && lone == 1 && bc > d && a.st.csize[bc] == 1) okm = 0;
      if constexpr (G > 32) {
        if (lane == 0) red_i[0] = okm;
        __syncthreads();
        mv = red_i[0];
      } else {
        mv = __shfl_sync(Grp<G>::mask(), okm, 0, G);
      }
    }
    if (!mv) continue;
    if (lane == 0) {
      if (a.fast) {
        atomic_add_a(&a.st.Sig[d], -ki);
        atomic_add_a(&a.st.Sig[bc], ki);
        atomicSub(&a.st.csize[d], 1);
        atomicAdd(&a.st.csize[bc], 1);
      } else {
        a.st.mv_from[i] = d;
        a.st.mv_to[i] = bc;
      }
      a.st.Cp[i] = bc;
      if (gcv) {
        if (M::is_fp) atomicAdd(&gcv->sum_f, (double)best);
        else atomic_add_u128(&gcv->sum_lo, &gcv->sum_hi, (unsigned long long)best, 0ULL);
      } else if (M::is_fp) {
        acc_f += (double)best;
      } else {
        const unsigned long long b = (unsigned long long)best;
        acc_lo += b;
        if (acc_lo < b) acc_hi++;
      }
      moved++;
    }
    if (a.pruning) {  // mark neighbours as unprocessed
#pragma unroll
      for (int x = 0; x < R; x++)
#pragma unroll
        for (int u = 0; u < U; u++) {
          const int e = lane + (x * U + u) * G;
          const int32_t j = R == 1 ? jj[u] : (e < deg ? rtg[e] : i);
          if (j != i) { a.st.flags[j] = 1; marks++; }
        }
    }
  }
  flush_move_acc<M::is_fp>(ctrl, acc_lo, acc_hi, moved, acc_f, r_lo, r_hi, r_mv, r_f);
  unsigned long long ctr[6] = {listed, processed, arcs, cand, moved, marks};
  block_add_counters<6, NW>(ctrl->lm_stat[a.bucket], ctr);
}

// Opts a kernel into more than 48 KB of dynamic shared memory, once per device (outside any graph
// capture: move_prepare runs it for every instantiation before an iteration is captured).
template <class M, class P>
static void lm_attr() {
  constexpr size_t smem = P::template smem<typename M::h_t>();
  if (smem <= 48 * 1024) return;
  static std::atomic<unsigned long long> done{0};  // one bit per device
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 64 && (done.load() >> dev) & 1ULL) return;
  cudaFuncSetAttribute(lm_kernel<M, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (dev < 64) done.fetch_or(1ULL << dev);
}

void move_prepare() {
  lm_attr<IntMode, Lm4>();
  lm_attr<IntMode, Lm5>();
  lm_attr<FpMode, Lm4>();
  lm_attr<FpMode, Lm5>();
}

template <class M, class P>
static void launch_lm(Ctx& c, const LmArgs<M>& a, int max_blocks) {
  lm_attr<M, P>();
  // device-resident range: a.count is then an upper bound of the range (a power of two)
  const int grid = grid_for(a.count, P::GPB, P::T < kBlock ? max_blocks * (kBlock / P::T) : max_blocks);
  lm_kernel<M, P><<<grid, P::T, P::template smem<typename M::h_t>(), c.s>>>(a);
  c.launches++;
}

template <class M>
void move_bucket(Ctx& c, int bucket, const GraphView<typename M::w_t>& g, const PassState<M>& st,
                 const int32_t* list, int64_t count, bool fast, bool pruning,
                 const int64_t* rng) {
  if (count <= 0 && !rng) return;
  LmArgs<M> a;
  a.g = g; a.st = st; a.list = list; a.count = count;
  a.rng = rng;
  a.fast = fast ? 1 : 0;
  a.pruning = pruning ? 1 : 0;
  a.bucket = bucket < kNumBuckets ? bucket : kNumBuckets - 1;
  a.tf = c.table_factor;
  const int cap = c.num_sms * c.lm_blocks_per_sm;
  switch (bucket) {
    case 0: launch_lm<M, Lm0>(c, a, cap); break;
    case 1: launch_lm<M, Lm1>(c, a, cap); break;
    case 2: launch_lm<M, Lm2>(c, a, cap); break;
    case 3: launch_lm<M, Lm3>(c, a, cap); break;
    case 4: launch_lm<M, Lm4>(c, a, cap); break;
    case 5: launch_lm<M, Lm5>(c, a, cap); break;
    default: break;  // giants go through giant_move
  }
}

// ---------------------------------------------------------------- deterministic apply
template <class M>
__global__ void lm_apply(PassState<M> st, const int32_t* list, int64_t count, const int64_t* rng) {
  if (*(volatile int32_t*)&st.ctrl->done) return;
  if (rng) {
    list += rng[0];
    count = rng[1];
  }
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < count; k += (int64_t)gridDim.x * blockDim.x) {
    const int32_t i = list[k];
    const int32_t t = st.mv_to[i];
    if (t >= 0) {
      const typename M::a_t ki = st.K[i];
      atomic_add_a(&st.Sig[st.mv_from[i]], -ki);
      atomic_add_a(&st.Sig[t], ki);
      st.mv_to[i] = -1;
    }
  }
}
template <class M>
void move_apply(Ctx& c, const PassState<M>& st, const int32_t* list, int64_t count, const int64_t* rng) {
  if (count <= 0 && !rng) return;
  const int grid = rng ? c.num_sms * 8 : grid_for(count, kBlock, c.num_sms * 8);
  lm_apply<M><<<grid, kBlock, 0, c.s>>>(st, list, count, rng);
  c.launches++;
}

// ---------------------------------------------------------------- iteration control
// Algorithm 2's tolerance test on the device: converged iff 2 sum N <= tau (2m)^2, with the
// 128-bit sum rounded once to double (integer mode) and the right side as tau * (t * t).
template <bool FP>
__global__ void lm_finish(Ctrl* c) {
  if (c->done) return;
  const int it = c->iterations + 1;
  c->iterations = it;
  bool conv;
  if (FP) {
    conv = __dmul_rn(2.0, c->sum_f) <= __dmul_rn(c->tau, __dmul_rn(c->two_m_f, c->two_m_f));
  } else {
    const unsigned long long hi = (c->sum_hi << 1) | (c->sum_lo >> 63), lo = c->sum_lo << 1;
    const double lhs = u128_to_double_rn(hi, lo);
    const double t = __ll2double_rn(c->two_m_i);
    conv = lhs <= __dmul_rn(c->tau, __dmul_rn(t, t));
  }
  c->moves_pass += c->moves;
  c->moves = 0;
  c->sum_lo = 0;
  c->sum_hi = 0;
  c->sum_f = 0.0;
  if (conv || it >= c->max_iterations) c->done = 1;
}
template <class M>
void move_finish(Ctx& c, Ctrl* ctrl) {
  lm_finish<M::is_fp><<<1, 1, 0, c.s>>>(ctrl);
  c.launches++;
}

__global__ void k_move_setup(Ctrl* c, double tau, int max_iterations) {
  c->done = max_iterations <= 0 ? 1 : 0;
  c->iterations = 0;
  c->max_iterations = max_iterations;
  c->tau = tau;
  c->sum_lo = 0;
  c->sum_hi = 0;
  c->sum_f = 0.0;
  c->moves = 0;
  c->moves_pass = 0;
}
void move_setup(Ctx& c, Ctrl* ctrl, double tau, int max_iterations) {
  k_move_setup<<<1, 1, 0, c.s>>>(ctrl, tau, max_iterations);
  c.launches++;
}

// ---------------------------------------------------------------- share of the arcs in hub rows
__global__ void k_hub_share(const int64_t* rbeg, const int64_t* rend, int64_t n, Ctrl* ctrl) {
  unsigned long long hub = 0, all = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const unsigned long long d = (unsigned long long)(rend[i] - rbeg[i]);
    all += d;
    if (d > 512) hub += d;
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    hub += __shfl_xor_sync(0xffffffffu, hub, o);
    all += __shfl_xor_sync(0xffffffffu, all, o);
  }
  if ((threadIdx.x & 31) == 0 && all) {
    atomicAdd(&ctrl->hub_arcs, hub);
    atomicAdd(&ctrl->all_arcs, all);
  }
}
template <class W>
void hub_share(Ctx& c, const GraphView<W>& g, Ctrl* ctrl) {
  cudaMemsetAsync(&ctrl->hub_arcs, 0, 2 * sizeof(unsigned long long), c.s);
  if (g.n <= 0) return;
  k_hub_share<<<grid_for(g.n, kBlock, c.num_sms * 8), kBlock, 0, c.s>>>(g.rbeg, g.rend, g.n, ctrl);
  c.launches++;
}
template void hub_share<int32_t>(Ctx&, const GraphView<int32_t>&, Ctrl*);
template void hub_share<float>(Ctx&, const GraphView<float>&, Ctrl*);

// ---------------------------------------------------------------- per-pass vertex state
template <class M>
__global__ void k_vertex_init(PassState<M> st, int64_t n, int from_k) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    st.Cp[i] = (int32_t)i;
    st.flags[i] = 1;
    st.csize[i] = 1;
    st.mv_to[i] = -1;
    if (from_k) {
      st.Sig[i] = st.K[i];
    } else {
      st.K[i] = 0;
      st.Sig[i] = 0;
    }
  }
}
template <class M>
void vertex_init(Ctx& c, const PassState<M>& st, int64_t n, bool from_k) {
  if (n <= 0) return;
  k_vertex_init<M><<<grid_for(n, kBlock, c.num_sms * 8), kBlock, 0, c.s>>>(st, n, from_k ? 1 : 0);
  c.launches++;
}

// K_i = sum of row weights (self-loop once), one group per vertex.
template <class M, int G>
__global__ void __launch_bounds__(kBlock) k_row_sums(GraphView<typename M::w_t> g, const int32_t* list, int64_t count,
                                                     typename M::a_t* K, typename M::a_t* Sig, typename M::a_t* K0) {
  typedef typename M::a_t A;
  __shared__ A red[32];
  constexpr int GPB = G <= 32 ? kBlock / G : 1;
  const int gib = G <= 32 ? (int)(threadIdx.x / G) : 0;
  const unsigned lane = Grp<G>::lane();
  for (int64_t idx = (int64_t)blockIdx.x * GPB + gib; idx < count; idx += (int64_t)gridDim.x * GPB) {
    const int32_t i = list[idx];
    A s = A(0);
    for (int64_t e = g.rbeg[i] + lane; e < g.rend[i]; e += G) s += (A)g.w[e];
    s = group_sum<G>(s, red);
    if (lane == 0) { K[i] = s; Sig[i] = s; if (K0) K0[i] = s; }
  }
}
template <class M>
void row_sums(Ctx& c, const GraphView<typename M::w_t>& g, const int32_t* perm, const int64_t* hb,
              typename M::a_t* K, typename M::a_t* Sig, typename M::a_t* K0) {
  const int cap = c.num_sms * 16;
  for (int b = 0; b < kNumBuckets; b++) {
    int64_t cnt = hb[b + 1] - hb[b];
    if (cnt <= 0) continue;
    const int32_t* l = perm + hb[b];
    switch (b) {
      case 0: k_row_sums<M, 4><<<grid_for(cnt, kBlock / 4, cap), kBlock, 0, c.s>>>(g, l, cnt, K, Sig, K0); break;
      case 1: k_row_sums<M, 8><<<grid_for(cnt, kBlock / 8, cap), kBlock, 0, c.s>>>(g, l, cnt, K, Sig, K0); break;
      case 2:
      case 3: k_row_sums<M, 32><<<grid_for(cnt, kBlock / 32, cap), kBlock, 0, c.s>>>(g, l, cnt, K, Sig, K0); break;
      default: k_row_sums<M, 256><<<grid_for(cnt, 1, cap), kBlock, 0, c.s>>>(g, l, cnt, K, Sig, K0); break;
    }
    c.launches++;
  }
}

template <class M>
__global__ void k_total(const typename M::a_t* K, int64_t n, Ctrl* ctrl) {
  typedef typename M::a_t A;
  __shared__ A red[32];
  A s = A(0);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) s += K[i];
  s = group_sum<kBlock>(s, red);
  if (threadIdx.x == 0) {
    if (M::is_fp) atomicAdd(&ctrl->two_m_f, (double)s);
    else atomic_add_a(&ctrl->two_m_i, (long long)s);
  }
}
template <class M>
void total_weight(Ctx& c, const typename M::a_t* K, int64_t n, Ctrl* ctrl) {
  if (n <= 0) return;
  k_total<M><<<grid_for(n, kBlock * 8, c.num_sms * 4), kBlock, 0, c.s>>>(K, n, ctrl);
  c.launches++;
}

#define LV_MOVE_INST(M)                                                                                           \
  template void vertex_init<M>(Ctx&, const PassState<M>&, int64_t, bool);                                        \
  template void row_sums<M>(Ctx&, const GraphView<M::w_t>&, const int32_t*, const int64_t*, M::a_t*, M::a_t*,    \
                            M::a_t*);                                                                            \
  template void total_weight<M>(Ctx&, const M::a_t*, int64_t, Ctrl*);                                            \
  template void move_bucket<M>(Ctx&, int, const GraphView<M::w_t>&, const PassState<M>&, const int32_t*, int64_t, \
                               bool, bool, const int64_t*);                                                      \
  template void move_apply<M>(Ctx&, const PassState<M>&, const int32_t*, int64_t, const int64_t*);               \
  template void move_finish<M>(Ctx&, Ctrl*);
LV_MOVE_INST(IntMode)
LV_MOVE_INST(FpMode)

}  // namespace lv
