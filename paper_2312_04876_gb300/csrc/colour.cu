// colour.cu -- Jones-Plassmann colouring for the deterministic (colour-synchronous) schedule.
//
// The paper cites ordering vertices by a graph colouring as one way to parallelise Louvain
// (Section 2).  Here: priority p(v) = hash3(seed, pass, v), u before v iff (p(u), u) > (p(v), v).
// A vertex is coloured once every higher-priority neighbour is, with the smallest colour none of
// them holds -- exactly greedy colouring in decreasing priority, whatever the round structure.
//
// Push form.  Every vertex keeps a counter of uncoloured higher-priority neighbour arcs and a bitmap
// of the colours its coloured higher-priority neighbours hold, floor(deg / 32) + 1 words at word
// floor(row start / 32) + v (rows start in increasing order, so the bitmaps do not overlap and no
// scan places them).  A round takes the ready list (counter 0): each vertex reads the first free
// bit of its bitmap as its colour (at most its degree, so larger colours need no bit), then pushes
// to every lower-priority neighbour -- sets the colour's bit and decrements the counter, appending
// the neighbours that reach zero to the next round's list.
//
// Everything runs in one persistent launch: the counters, then one round per barrier.  What bounds
// it: wide rounds (first rounds of a low-degree graph) wait on gathers of the neighbours' records,
// narrow rounds (a dense core of k hubs needs k rounds: greedy colouring is sequential along
// priority chains) on the barrier and one chain of dependent loads.  So
//   * a list entry is a chunk of a row, not a row: the vertex that makes u ready appends all of u's
//     chunks, every chunk finds u's colour itself (one or two bitmap reads) and pushes its own arcs,
//     and a hub's push is spread over the GPU in the round that colours it, with one barrier a round;
//   * an entry of a wide round takes a few lanes with four arcs each; in a narrow round (a group of
//     one lane per arc for every entry) its accesses are one deep; it carries its arc range, so its
//     arcs, prefetched to L2 when it was appended, and its bitmap are loaded at once;
//   * a neighbour's counter, degree and row start are one 16-byte record: one gather per arc;
//   * a block keeps the short rows it makes ready in shared memory and takes them itself in the next
//     round; long rows and what does not fit go to a list in global memory (queued per warp, one
//     atomic per 32 entries);
//   * the launch takes the smallest scope that holds the graph (persist.cuh), and the size of the
//     next round comes with the barrier.
// R-MAT 22, pass 0 (128M arcs, 2,915 rounds): 17.2 ms, 5.9 us a round (a warp per row, two barriers a
// round: 42.9 ms); 24M-vertex grid, pass 0 (17 rounds): 6.2 ms (31.8 ms).
#include "persist.cuh"

namespace lv {

struct JpArgs {
  GraphView<int32_t> g;
  uint64_t key;                 // hash3 state after seed and pass: prio(v) = mix64(key + local id)
  int32_t* colour;
  int4* rec;                    // [n] {uncoloured higher-priority arcs, degree, row start (64 bits)}
  int4* lists[2];               // ready lists of JpEntry
  int64_t list_cap;
  unsigned* used;               // the bitmaps
  unsigned long long* st;       // kJp* below
  const int32_t* perm;          // vertices by degree bucket
  int32_t hb[kNumBuckets + 1];  // bucket offsets in perm
  Ctrl* ctrl;
  Segs seg;                     // batched run: priorities hash graph-local ids
};
// words of the colouring's state block (zeroed before the launch)
enum { kJpCount = 0 /* 3 rotating list sizes */, kJpBar = 3 /* 3 barrier words */, kJpColoured = 6, kJpColours,
       kJpRounds, kJpTrips, kJpWords };
static_assert(kJpWords <= kJpStateWords, "state block");

constexpr int kPersistThreads = 1024;
// CH, the arcs of a list entry: 8 on low-degree graphs, else 32.
constexpr int kJpQueue = 64;                          // queue slots of a warp (flushed from 32 on)
// Entries a block keeps for itself, of rows of at most kJpKeep chunks.  With several blocks only a
// narrow round's: what blocks keep drifts to a few of them (planted partition of 100,003 vertices,
// pass 0: 0.49 ms with 16, 0.66 with 96, 1.6 with 1024).
constexpr int kJpLocal = 1024, kJpLocalShared = 16, kJpKeep = 4;
constexpr size_t kJpSmem = sizeof(int4) * (2 * kJpLocal + (kPersistThreads / 32) * kJpQueue);
// What a block publishes with a barrier: its entries in the global list (bits 0-39) and whether it
// holds local ones (bits 40-51; a grid has far fewer than 4096 blocks).
constexpr int kJpLocalShift = 40;

// A list entry as one 16-byte word: vertex, degree, first arc (38 bits) and chunk index (26 bits: a
// row holds fewer than 2^31 arcs).
__device__ __forceinline__ int4 jp_entry(int32_t v, int deg, int64_t beg, int chunk, int ch) {
  const unsigned long long x = (unsigned long long)(beg + (int64_t)chunk * ch) | ((unsigned long long)chunk << 38);
  return make_int4(v, deg, (int)(unsigned)x, (int)(unsigned)(x >> 32));
}
__device__ __forceinline__ int64_t rec_beg(const int4& r) {
  return (int64_t)((unsigned long long)(unsigned)r.z | ((unsigned long long)(unsigned)r.w << 32));
}
__device__ __forceinline__ unsigned bitmap_word(int64_t beg, int32_t v) { return (unsigned)(beg >> 5) + (unsigned)v; }

// Predicated accesses: under a branch each would wait for its own result before the next is issued.
__device__ __forceinline__ int dec_if(bool p, int* addr) {  // old value, 0 if !p
  int old;
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %1, 0;\n\tmov.s32 %0, 0;\n\t@q atom.global.add.s32 %0, [%2], -1;\n\t}"
               : "=&r"(old) : "r"((int)p), "l"(addr) : "memory");
  return old;
}
__device__ __forceinline__ int4 load_if(bool p, const int4* addr) {
  int4 r;
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %4, 0;\n\tmov.s32 %0, 0;\n\tmov.s32 %1, 0;\n\tmov.s32 %2, 0;\n\tmov.s32 %3, 0;\n\t"
               "@q ld.global.v4.s32 {%0, %1, %2, %3}, [%5];\n\t}"
               : "=&r"(r.x), "=&r"(r.y), "=&r"(r.z), "=&r"(r.w) : "r"((int)p), "l"(addr) : "memory");
  return r;
}

// Where the vertices made ready in a round go.
struct JpOut {
  int cap;                    // entries the block keeps
  int4* local;                // this block's entries of the next round
  int* nlocal;                // their number (may pass kJpLocal: those went to the list)
  int* nglobal;               // entries this block appended to the list
  int4* list;                 // the next round's list and its size
  unsigned long long* count;
  int4* queue;                // this warp's queue for the list
};

__device__ __forceinline__ uint64_t jp_base(const JpArgs& a, int32_t v) {
  return a.seg.vg ? a.key - (uint64_t)a.seg.gc[a.seg.vg[v]].vbase : a.key;
}

// Appends entries [0, k) made by `make(t)` to the next list with one atomic.
template <class F>
__device__ __forceinline__ void jp_append(const JpArgs& a, const JpOut& o, int k, F make) {
  const int lane = threadIdx.x & 31;
  unsigned long long base = 0;
  if (lane == 0) {
    base = atomicAdd(o.count, (unsigned long long)k);
    atomicAdd(o.nglobal, k);
  }
  base = __shfl_sync(0xffffffffu, base, 0);
  for (int t = lane; t < k; t += 32) {
    if ((int64_t)(base + t) < a.list_cap) o.list[base + t] = make(t);
    else atomicAdd(&a.st[kJpTrips], 1ULL);
  }
}

__device__ __forceinline__ int lanes_scan(int x) {  // inclusive
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) >= o) x += y;
  }
  return x;
}

// Puts the lanes' ready vertices (U a lane) where they go.  All lanes of the warp call it.
template <int CH, int U>
__device__ __forceinline__ void jp_emit(const JpArgs& a, const JpOut& o, int& qn, const bool (&rdy)[U],
                                        const int32_t (&u)[U], const int4 (&rec)[U]) {
  const int lane = threadIdx.x & 31;
  int nloc = 0, nbig = 0;
#pragma unroll
  for (int x = 0; x < U; x++) {
    const int nch = (rec[x].y + CH - 1) / CH;
    if (rdy[x]) {
      if (nch <= kJpKeep) nloc += nch;
      else nbig += nch;
    }
  }
  if (!__any_sync(0xffffffffu, nloc + nbig > 0)) return;
  // short rows: this block's own entries while they fit
  bool over[U];
#pragma unroll
  for (int x = 0; x < U; x++) over[x] = false;
  if (__any_sync(0xffffffffu, nloc > 0)) {
    const int incl = lanes_scan(nloc);
    int base = 0;
    if (lane == 31) base = *(volatile int*)o.nlocal < o.cap ? atomicAdd(o.nlocal, incl) : o.cap;
    int slot = __shfl_sync(0xffffffffu, base, 31) + incl - nloc;
    bool any_over = false;
#pragma unroll
    for (int x = 0; x < U; x++) {
      const int nch = (rec[x].y + CH - 1) / CH;
      if (!rdy[x] || nch > kJpKeep) continue;
      over[x] = slot + nch > o.cap;
      any_over |= over[x];
      if (!over[x]) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.g.tg + rec_beg(rec[x])));
      for (int t = 0; t < nch; t++)
        if (!over[x]) o.local[slot + t] = jp_entry(u[x], rec[x].y, rec_beg(rec[x]), t, CH);
        else if (slot + t < o.cap) o.local[slot + t] = make_int4(0, 0, 0, 0);  // a hole: no arcs, no vertex
      slot += nch;
    }
    if (__any_sync(0xffffffffu, any_over)) {
#pragma unroll
      for (int x = 0; x < U; x++) {
        const bool one = over[x] && rec[x].y <= CH;
        const unsigned ob = __ballot_sync(0xffffffffu, one);
        if (one) o.queue[qn + __popc(ob & lanemask_lt())] = jp_entry(u[x], rec[x].y, rec_beg(rec[x]), 0, CH);
        qn += __popc(ob);
        __syncwarp();
        if (qn >= 32) {
          jp_append(a, o, qn, [&](int t) { return o.queue[t]; });
          qn = 0;
          __syncwarp();
        }
        if (over[x] && rec[x].y > CH) nbig += (rec[x].y + CH - 1) / CH;
      }
    }
  }
  // long rows, and rows of several chunks that did not fit: the global list, one reservation
  if (__any_sync(0xffffffffu, nbig > 0)) {
    const int incl = lanes_scan(nbig);
    unsigned long long base = 0;
    if (lane == 31) {
      base = atomicAdd(o.count, (unsigned long long)incl);
      atomicAdd(o.nglobal, incl);
    }
    unsigned long long at = __shfl_sync(0xffffffffu, base, 31) + (unsigned long long)(incl - nbig);
#pragma unroll
    for (int x = 0; x < U; x++) {
      const int nch = (rec[x].y + CH - 1) / CH;
      const bool big = rdy[x] && (nch > kJpKeep || (over[x] && nch > 1));
      for (unsigned m = __ballot_sync(0xffffffffu, big); m; m &= m - 1) {
        const int src = __ffs(m) - 1;
        const int32_t bu = __shfl_sync(0xffffffffu, u[x], src);
        const int bd = __shfl_sync(0xffffffffu, rec[x].y, src);
        const int64_t bb = __shfl_sync(0xffffffffu, rec_beg(rec[x]), src);
        const unsigned long long b0 = __shfl_sync(0xffffffffu, at, src);
        for (int t = lane; t < (bd + CH - 1) / CH; t += 32) {
          asm volatile("prefetch.global.L2 [%0];" ::"l"(a.g.tg + bb + (int64_t)t * CH));
          if ((int64_t)(b0 + t) < a.list_cap) o.list[b0 + t] = jp_entry(bu, bd, bb, t, CH);
          else atomicAdd(&a.st[kJpTrips], 1ULL);
        }
      }
      if (big) at += (unsigned long long)nch;
    }
  }
}

// Counters, records and cleared bitmaps of the vertices list[0, count), G lanes a row (G <= 32), and
// the first ready list.
template <int CH, int G>
__device__ __forceinline__ void jp_count(const JpArgs& a, const int32_t* list, int64_t count, const JpOut& o, int& qn) {
  constexpr int U = 4, GPW = 32 / G;
  const int lane = threadIdx.x & 31, gl = lane & (G - 1);
  const int64_t nw = (int64_t)gridDim.x * (kPersistThreads / 32);
  for (int64_t t0 = ((int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * GPW; t0 < count; t0 += nw * GPW) {
    const int64_t idx = t0 + lane / G;
    const bool on = idx < count;
    int32_t v = 0, k = 0;
    int64_t beg = 0, end = 0;
    uint64_t pv = 0, base = 0;
    if (on) {
      v = list[idx];
      beg = a.g.rbeg[v];
      end = a.g.rend[v];
      base = jp_base(a, v);
      pv = mix64(base + (uint64_t)v);
    }
    for (int64_t e0 = beg + gl; e0 < end; e0 += G * U) {
      int32_t uu[U];
#pragma unroll
      for (int x = 0; x < U; x++) uu[x] = e0 + x * G < end ? a.g.tg[e0 + x * G] : v;
#pragma unroll
      for (int x = 0; x < U; x++)
        if (uu[x] != v && higher(mix64(base + (uint64_t)uu[x]), uu[x], pv, v)) k++;
    }
    __syncwarp();
#pragma unroll
    for (int x = G / 2; x >= 1; x >>= 1) k += __shfl_xor_sync(0xffffffffu, k, x);
    const int deg = (int)(end - beg);
    if (on) {
      const unsigned w0 = bitmap_word(beg, v);
      for (int w = gl; w <= deg >> 5; w += G) a.used[w0 + w] = 0u;
      if (gl == 0) a.rec[v] = make_int4(k, deg, (int)(unsigned)beg, (int)(beg >> 32));
    }
    const bool rdy[1] = {on && gl == 0 && k == 0};
    const int32_t rv[1] = {v};
    const int4 rr[1] = {make_int4(k, deg, (int)(unsigned)beg, (int)(beg >> 32))};
    jp_emit<CH, 1>(a, o, qn, rdy, rv, rr);
  }
}

// The same for long rows, one block a row.
template <int CH>
__device__ __forceinline__ void jp_count_rows(const JpArgs& a, const int32_t* list, int64_t count, const JpOut& o,
                                              int& qn) {
  constexpr int U = 4;
  __shared__ int s_k;
  for (int64_t idx = blockIdx.x; idx < count; idx += gridDim.x) {
    const int32_t v = list[idx];
    const int64_t beg = a.g.rbeg[v], end = a.g.rend[v];
    const uint64_t base = jp_base(a, v), pv = mix64(base + (uint64_t)v);
    if (threadIdx.x == 0) s_k = 0;
    __syncthreads();
    int k = 0;
    for (int64_t e0 = beg + threadIdx.x; e0 < end; e0 += kPersistThreads * U) {
      int32_t uu[U];
#pragma unroll
      for (int x = 0; x < U; x++) uu[x] = e0 + x * kPersistThreads < end ? a.g.tg[e0 + x * kPersistThreads] : v;
#pragma unroll
      for (int x = 0; x < U; x++)
        if (uu[x] != v && higher(mix64(base + (uint64_t)uu[x]), uu[x], pv, v)) k++;
    }
    __syncwarp();
#pragma unroll
    for (int x = 16; x >= 1; x >>= 1) k += __shfl_xor_sync(0xffffffffu, k, x);
    if ((threadIdx.x & 31) == 0 && k) atomicAdd(&s_k, k);
    const int deg = (int)(end - beg);
    const unsigned w0 = bitmap_word(beg, v);
    for (int w = threadIdx.x; w <= deg >> 5; w += kPersistThreads) a.used[w0 + w] = 0u;
    __syncthreads();
    if (threadIdx.x < 32) {
      k = s_k;
      if (threadIdx.x == 0) a.rec[v] = make_int4(k, deg, (int)(unsigned)beg, (int)(beg >> 32));
      const bool rdy[1] = {threadIdx.x == 0 && k == 0};
      const int32_t rv[1] = {v};
      const int4 rr[1] = {make_int4(k, deg, (int)(unsigned)beg, (int)(beg >> 32))};
      jp_emit<CH, 1>(a, o, qn, rdy, rv, rr);
    }
    __syncthreads();
  }
}

// What a thread's entries coloured.
struct JpDone {
  unsigned long long coloured;
  int colours;
};

// Entries in[0, n) of a round, CH / U lanes each; groups first, first + step, ... of the entries' order
// are this warp's (`first` in groups of one warp).
template <int CH, int U>
__device__ __forceinline__ void jp_entries(const JpArgs& a, const JpOut& o, int& qn, JpDone& done, const int4* in,
                                           int64_t n, int64_t first, int64_t step) {
  constexpr int L = CH / U, GPW = 32 / L;
  const int lane = threadIdx.x & 31, gl = lane & (L - 1);
  for (int64_t t0 = first * GPW; t0 < n; t0 += step * GPW) {
    const int64_t idx = t0 + lane / L;
    const int4 en = idx < n ? in[idx] : make_int4(0, 0, 0, 0);
    const bool on = en.y > 0;
    const int32_t v = en.x;
    const int chunk = (int)((unsigned)en.w >> 6);
    const int64_t start = (int64_t)((unsigned long long)(unsigned)en.z | ((unsigned long long)((unsigned)en.w & 63u) << 32));
    const uint64_t base = on ? jp_base(a, v) : 0;
    // this chunk's targets are loaded while the bitmap is read
    const int e0 = chunk * CH + gl;
    int32_t uu[U];
#pragma unroll
    for (int x = 0; x < U; x++) uu[x] = e0 + x * L < en.y ? a.g.tg[start + gl + x * L] : v;
    // first free bit; it exists: the colours recorded number at most the degree
    const unsigned bw = bitmap_word(start - (int64_t)chunk * CH, v);
    const int words = on ? (en.y >> 5) + 1 : 0;
    int col = -1;
    for (int wb = 0; __any_sync(0xffffffffu, col < 0 && wb < words); wb += L) {
      const unsigned freeb = wb + gl < words ? ~a.used[bw + wb + gl] : 0u;
      const unsigned ball = (__ballot_sync(0xffffffffu, freeb != 0u) >> (lane & ~(L - 1))) & (0xffffffffu >> (32 - L));
      const int f = ball ? __ffs(ball) - 1 : 0;
      const unsigned fw = __shfl_sync(0xffffffffu, freeb, f, L);
      if (col < 0 && ball) col = 32 * (wb + f) + __ffs(fw) - 1;
    }
    if (on && col < 0) {  // unreachable
      atomicOr(&a.ctrl->error, kErrRange);
      col = 0;
    }
    if (on && chunk == 0 && gl == 0) {
      a.colour[v] = col;
      done.coloured++;
      if (col >= done.colours) done.colours = col + 1;
    }
    // push to the lower-priority neighbours: the counter is decremented while the rest of the
    // record is read; a neighbour that becomes ready is taken after the barrier, which orders the
    // bit before that
    const uint64_t pv = mix64(base + (uint64_t)v);
    bool low[U], rdy[U];
    int left[U];
    int4 ru[U];
#pragma unroll
    for (int x = 0; x < U; x++) low[x] = uu[x] != v && higher(pv, v, mix64(base + (uint64_t)uu[x]), uu[x]);
#pragma unroll
    for (int x = 0; x < U; x++) left[x] = dec_if(low[x], &a.rec[uu[x]].x);
#pragma unroll
    for (int x = 0; x < U; x++) ru[x] = load_if(low[x], &a.rec[uu[x]]);
#pragma unroll
    for (int x = 0; x < U; x++) rdy[x] = left[x] == 1;
#pragma unroll
    for (int x = 0; x < U; x++)
      if (low[x] && (col >> 5) <= (ru[x].y >> 5))
        atomicOr(&a.used[bitmap_word(rec_beg(ru[x]), uu[x]) + (col >> 5)], 1u << (col & 31));
    jp_emit<CH, U>(a, o, qn, rdy, uu, ru);
  }
}

template <int SC, int CH>
__global__ void __launch_bounds__(kPersistThreads, 1) jp_persistent(JpArgs a, PersistBar bar) {
  extern __shared__ __align__(16) unsigned char jp_dyn[];  // two local lists, the warps' queues
  constexpr int kWarps = kPersistThreads / 32;
  constexpr int64_t kGroups = kWarps * (32 / CH);  // one-lane-per-arc groups of a block
  __shared__ int s_nlocal[3], s_nglobal[3];  // of the list filled before barrier r, at r % 3
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int4* const local = reinterpret_cast<int4*>(jp_dyn);
  JpOut o;
  o.cap = SC == kCta ? kJpLocal : kJpLocalShared;
  o.queue = local + 2 * kJpLocal + warp * kJpQueue;
  int qn = 0;
  if (threadIdx.x < 3) { s_nlocal[threadIdx.x] = 0; s_nglobal[threadIdx.x] = 0; }
  __syncthreads();
  JpDone done = {0, 0};
  int64_t n = 0;  // entries of the global list
  // round r takes the list that barrier r completed and fills the next one
  for (unsigned r = 0;; r++) {
    o.local = local + (r & 1) * kJpLocal;
    o.nlocal = &s_nlocal[r % 3];
    o.nglobal = &s_nglobal[r % 3];
    o.list = a.lists[r & 1];
    o.count = &a.st[kJpCount + r % 3];
    if (r == 0) {
      jp_count<CH, 1>(a, a.perm + a.hb[0], a.hb[1] - a.hb[0], o, qn);
      jp_count<CH, 4>(a, a.perm + a.hb[1], a.hb[2] - a.hb[1], o, qn);
      // rows of 513-2048 arcs: a warp each where they are many, else a block each like the longer ones
      const int long0 = a.hb[5] - a.hb[4] > 8 * (int)gridDim.x ? 5 : 4;
      jp_count<CH, 32>(a, a.perm + a.hb[2], a.hb[long0] - a.hb[2], o, qn);
      jp_count_rows<CH>(a, a.perm + a.hb[long0], a.hb[kNumBuckets] - a.hb[long0], o, qn);
    } else {
      // the list of round r - 1's barrier: this block's entries from its last warp down (the first warps
      // have the global list's), then its share of the global list, whose consecutive entries go to
      // different blocks
      const int4* lin = local + ((r - 1) & 1) * kJpLocal;
      const int nl = min(s_nlocal[(r - 1) % 3], o.cap);
      if (nl <= kGroups) jp_entries<CH, 1>(a, o, qn, done, lin, nl, kWarps - 1 - warp, kWarps);
      else jp_entries<CH, 4>(a, o, qn, done, lin, nl, kWarps - 1 - warp, kWarps);
      const int4* in = a.lists[(r - 1) & 1];
      const int64_t first = (int64_t)warp * gridDim.x + blockIdx.x, step = (int64_t)gridDim.x * kWarps;
      if (n <= kGroups * gridDim.x) jp_entries<CH, 1>(a, o, qn, done, in, n, first, step);
      else jp_entries<CH, 4>(a, o, qn, done, in, n, first, step);
    }
    if (qn) jp_append(a, o, qn, [&](int t) { return o.queue[t]; });
    qn = 0;
    unsigned long long sum = 0;
    const bool ok = scope_barrier<SC>(bar, a.ctrl, &sum, [&]() {
      return (unsigned long long)*(volatile int*)o.nglobal |
             ((unsigned long long)(*(volatile int*)o.nlocal > 0) << kJpLocalShift);
    });
    sum &= kBarSum;
    if (!ok || sum == 0) break;  // a wait ran out, or nothing is ready: every listed vertex is coloured
    n = (int64_t)(sum & ((1ULL << kJpLocalShift) - 1));
    if (n > a.list_cap) n = a.list_cap;
    if (threadIdx.x == 0) {  // the counters that the round after next fills; last read before this barrier
      s_nlocal[(r + 2) % 3] = 0;
      s_nglobal[(r + 2) % 3] = 0;
      if (blockIdx.x == 0) {
        a.st[kJpCount + (r + 2) % 3] = 0;
        a.st[kJpRounds] = r + 1;
      }
    }
  }
  unsigned long long coloured = done.coloured;
  int colours = done.colours;
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    coloured += __shfl_xor_sync(0xffffffffu, coloured, o);
    colours = max(colours, __shfl_xor_sync(0xffffffffu, colours, o));
  }
  if (lane == 0 && coloured) {
    atomicAdd(&a.st[kJpColoured], coloured);
    atomicMax(&a.st[kJpColours], (unsigned long long)colours);
  }
}

template <int CH>
static cudaError_t jp_launch(Scope sc, const Ctx& c, const JpArgs& a, const PersistBar& bar) {
  if (sc == kCta) return scope_launch(sc, c, jp_persistent<kCta, CH>, kPersistThreads, kJpSmem, a, bar);
  if (sc == kCluster) return scope_launch(sc, c, jp_persistent<kCluster, CH>, kPersistThreads, kJpSmem, a, bar);
  return scope_launch(sc, c, jp_persistent<kGrid, CH>, kPersistThreads, kJpSmem, a, bar);
}

int32_t jp_colour(Ctx& c, const GraphView<int32_t>& g, const int32_t* perm, const int64_t* hb, uint64_t seed,
                  int32_t pass, int32_t* colour, const JpBuffers& jb, Ctrl* ctrl, unsigned long long* h_pinned,
                  cudaError_t* err, int64_t giant_arcs, Segs seg, int64_t* rounds_out) {
  const int64_t listed = hb[kNumBuckets] - hb[0];
  if (listed < g.n) fill_i32(c, colour, 0, g.n);  // isolated vertices (not listed) get colour 0
  if ((*err = cudaMemsetAsync(jb.state, 0, kJpWords * sizeof(unsigned long long), c.s)) != cudaSuccess) return -1;
  JpArgs a;
  a.g = g; a.colour = colour; a.rec = jb.rec; a.lists[0] = jb.list0; a.lists[1] = jb.list1; a.list_cap = jb.list_cap;
  a.used = jb.used; a.st = jb.state; a.perm = perm; a.ctrl = ctrl; a.seg = seg;
  // hash3(seed, pass, v) = mix64(key + v)
  const uint64_t gm = 0x9e3779b97f4a7c15ULL;
  a.key = mix64(mix64(seed + gm) + (uint64_t)pass + 2 * gm) + 3 * gm;
  for (int b = 0; b <= kNumBuckets; b++) a.hb[b] = (int32_t)hb[b];
  PersistBar bar{jb.state + kJpBar, c.wait_spins > 0 ? c.wait_spins : kBarrierPolls, 0, 0};
  // entries a round may hold at most with 8-arc chunks, and the arcs, about
  static const int64_t kChunks[kNumBuckets] = {1, 2, 16, 64, 256, 512, 0};
  int64_t chunks = 0, arcs = 0;
  for (int b = 0; b < kNumBuckets; b++) {
    chunks += (hb[b + 1] - hb[b]) * kChunks[b];
    const int64_t about = (hb[b + 1] - hb[b]) * kTypicalArcs[b];
    arcs += b == kNumBuckets - 1 && giant_arcs > about ? giant_arcs : about;
  }
  const bool low = hb[kNumBuckets] == hb[kNumBuckets - 1] && chunks <= jb.list_cap && arcs <= 8 * listed;
  // One block up to ~60,000 arcs, a cluster up to ~500,000 arcs on few vertices (dense super-vertex
  // graphs: many narrow rounds), else the grid.  Measured: 99 vertices, 9,741 arcs, 99 rounds 0.24 ms
  // on a block, 0.42 on the grid; 199 vertices, 18,126 arcs 0.31 against 0.45 on a cluster; 2,855
  // vertices, 255,755 arcs, 492 rounds 1.69 ms on a cluster, 2.14 on the grid; 10,000 vertices,
  // 143,254 arcs, 35 rounds 0.32 on a cluster, 0.27 on the grid.  A caller that bounds the waits
  // (params.wait_spins) gets the grid's bounded barrier.
  Scope sc = kGrid;
  if (c.wait_spins <= 0 && arcs <= 60000) sc = kCta;
  else if (c.wait_spins <= 0 && arcs <= 524288 && listed <= 8192) sc = kCluster;
  *err = low ? jp_launch<8>(sc, c, a, bar) : jp_launch<32>(sc, c, a, bar);
  if (*err != cudaSuccess && sc != kCta) {  // the scope cannot be launched here: one block can
    cudaGetLastError();
    *err = low ? jp_launch<8>(kCta, c, a, bar) : jp_launch<32>(kCta, c, a, bar);
  }
  c.launches++;
  if (*err != cudaSuccess) return -1;
  cudaMemcpyAsync(h_pinned, jb.state, kJpWords * sizeof(unsigned long long), cudaMemcpyDeviceToHost, c.s);
  if ((*err = cudaStreamSynchronize(c.s)) != cudaSuccess) return -1;
  if ((int64_t)h_pinned[kJpColoured] != listed || h_pinned[kJpTrips]) {
    const unsigned long long q[5] = {h_pinned[kJpColoured], h_pinned[kJpColours], (unsigned long long)listed,
                                     h_pinned[kJpRounds], h_pinned[kJpTrips]};
    for (int k = 0; k < 5; k++) h_pinned[3 + k] = q[k];
    return -1;
  }
  if (rounds_out) *rounds_out = (int64_t)h_pinned[kJpRounds];
  const int32_t ncol = (int32_t)h_pinned[kJpColours];
  return ncol > 0 ? ncol : 1;
}

}  // namespace lv
