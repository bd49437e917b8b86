// validate.cu -- input checks of the CSR contract (Section 3: an undirected weighted graph,
// w_ij = w_ji > 0, stored with both arcs).  Offsets are checked first (the arc checks trust
// them); then targets, weights, the weight total (2m) and symmetry.  Symmetry is tested by a
// signed hash sum: every arc (u -> v, w), u != v, adds +h(min, max, w) if u < v and -h if u > v,
// modulo 2^64, so a symmetric arc multiset sums to zero and any other fails with probability
// 1 - 2^-64.  Results land in ctrl counters; the host turns them into LOUVAIN_ERR_INVALID.
#include "internal.cuh"

namespace lv {

__global__ void k_val_offsets(int64_t n, int64_t n_arcs, const int64_t* offs, Ctrl* ctrl) {
  unsigned long long bad = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    if (offs[i + 1] < offs[i]) bad++;
  if (blockIdx.x == 0 && threadIdx.x == 0 && (offs[0] != 0 || offs[n] != n_arcs)) bad++;
  if (bad) atomicAdd(&ctrl->cnt[0], bad);
}

void validate_offsets(Ctx& c, int64_t n, int64_t n_arcs, const int64_t* offs, Ctrl* ctrl) {
  k_val_offsets<<<grid_for(n > 0 ? n : 1, kBlock, c.num_sms * 8), kBlock, 0, c.s>>>(n, n_arcs, offs, ctrl);
  c.launches++;
}

// Last row r in [lo, hi) with offs[r] <= e, for an arc e of [offs[lo], offs[hi]).
__device__ __forceinline__ int64_t val_row(const int64_t* offs, int64_t lo, int64_t hi, int64_t e) {
  while (hi - lo > 1) {
    const int64_t mid = (lo + hi) >> 1;
    if (offs[mid] <= e) lo = mid; else hi = mid;
  }
  return lo;
}

// A warp checks a contiguous range of arcs: one binary search finds its first row, then the ends of the
// next 32 rows, one a lane, give every lane its arc's row by shuffles (a longer run of short or empty
// rows falls back to the search).  By arcs and not by rows because rows are not alike: with 256 rows a
// block, the blocks of R-MAT 20's hubs took 4.2 ms for arcs whose bytes take 0.04 (a modularity and an
// aggregation on that graph with fp32 weights, both validating: 10.7 -> 3.5 ms).  What bounds it now is the
// 64-bit hash of an arc.
template <bool FP>
__global__ void __launch_bounds__(kBlock) k_val_arcs(int64_t n, const int64_t* offs, const int32_t* tg, const void* wv,
                                                     Ctrl* ctrl) {
  unsigned long long bad_t = 0, bad_w = 0, sym = 0, isum = 0;
  double fsum = 0.0;
  constexpr int U = 4;
  const int lane = threadIdx.x & 31;
  const int64_t arcs = offs[n], warps = (int64_t)gridDim.x * (kBlock / 32);
  const int64_t span = ((arcs + warps - 1) / warps + 32 * U - 1) / (32 * U) * (32 * U);
  const int64_t a0 = ((int64_t)blockIdx.x * (kBlock / 32) + (threadIdx.x >> 5)) * span;
  const int64_t a1 = a0 + span < arcs ? a0 + span : arcs;
  int64_t r = a0 < a1 ? val_row(offs, 0, n, a0) : 0;  // row of the first arc of a step
  for (int64_t base = a0; base < a1; base += 32 * U) {
    int32_t vv[U];
    uint32_t ww[U];
#pragma unroll
    for (int x = 0; x < U; x++) {
      const int64_t e = base + x * 32 + lane;
      vv[x] = e < a1 ? tg[e] : 0;
      ww[x] = e < a1 ? reinterpret_cast<const uint32_t*>(wv)[e] : 0u;
    }
#pragma unroll
    for (int x = 0; x < U; x++) {
      const int64_t e = base + x * 32 + lane;
      if (base + x * 32 >= a1) break;  // uniform
      // rows whose end is at most e, counted among rows r .. r + 31
      const int64_t end = offs[r + 1 + lane < n ? r + 1 + lane : n];
      int c = 0;
#pragma unroll
      for (int step = 16; step >= 1; step >>= 1)
        if (__shfl_sync(0xffffffffu, end, c + step - 1) <= e) c += step;
      int64_t u = r + c;
      if (__shfl_sync(0xffffffffu, end, 31) <= e && e < a1) u = val_row(offs, r, n, e);
      r = __shfl_sync(0xffffffffu, u, (int)(a1 - 1 - (base + x * 32) < 31 ? a1 - 1 - (base + x * 32) : 31));
      if (e >= a1) continue;
      const int32_t v = vv[x];
      if (FP) {
        const float w = __uint_as_float(ww[x]);
        if (!(w > 0.0f) || isinf(w)) bad_w++;
        else fsum += (double)w;
      } else {
        const int32_t w = (int32_t)ww[x];
        if (w <= 0) bad_w++;
        else isum += (unsigned long long)w;
      }
      if (v < 0 || v >= n) { bad_t++; continue; }
      if (v == u) continue;
      const int64_t lo = u < v ? u : v, hi = u < v ? v : u;
      const uint64_t h = hash3(0x5EEDULL, ((uint64_t)lo << 32) | (uint64_t)hi, ww[x]);
      sym += u < v ? h : (0ULL - h);
    }
  }
  __syncwarp();
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    bad_t += __shfl_xor_sync(0xffffffffu, bad_t, o);
    bad_w += __shfl_xor_sync(0xffffffffu, bad_w, o);
    sym += __shfl_xor_sync(0xffffffffu, sym, o);
    isum += __shfl_xor_sync(0xffffffffu, isum, o);
    fsum += __shfl_xor_sync(0xffffffffu, fsum, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (bad_t) atomicAdd(&ctrl->cnt[1], bad_t);
    if (bad_w) atomicAdd(&ctrl->cnt[2], bad_w);
    if (sym) atomicAdd(&ctrl->cnt[3], sym);
    if (isum) atomicAdd(reinterpret_cast<unsigned long long*>(&ctrl->acc_i[0]), isum);
    if (fsum != 0.0) atomicAdd(&ctrl->acc_f[0], fsum);
  }
}

void validate_arcs(Ctx& c, int64_t n, int64_t n_arcs, const int64_t* offs, const int32_t* tg, const void* w, bool fp,
                   Ctrl* ctrl) {
  if (n <= 0) return;
  const int grid = grid_for(n_arcs, kBlock * 4, c.num_sms * 8);
  if (fp) k_val_arcs<true><<<grid, kBlock, 0, c.s>>>(n, offs, tg, w, ctrl);
  else k_val_arcs<false><<<grid, kBlock, 0, c.s>>>(n, offs, tg, w, ctrl);
  c.launches++;
}

__global__ void k_val_range(const int32_t* ids, int64_t m, int64_t hi, Ctrl* ctrl) {
  unsigned long long bad = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
    if (ids[i] < 0 || ids[i] >= hi) bad++;
  if (bad) atomicAdd(&ctrl->cnt[5], bad);
}

void validate_range(Ctx& c, const int32_t* ids, int64_t m, int64_t hi, Ctrl* ctrl) {
  if (m <= 0) return;
  k_val_range<<<grid_for(m, kBlock, c.num_sms * 8), kBlock, 0, c.s>>>(ids, m, hi, ctrl);
  c.launches++;
}

__global__ void k_val_reset(Ctrl* c) {
  for (int k = 0; k < 8; k++) c->cnt[k] = 0;
  for (int k = 0; k < 4; k++) { c->acc_i[k] = 0; c->acc_f[k] = 0.0; }
}
void validate_reset(Ctx& c, Ctrl* ctrl) {
  k_val_reset<<<1, 1, 0, c.s>>>(ctrl);
  c.launches++;
}

}  // namespace lv
