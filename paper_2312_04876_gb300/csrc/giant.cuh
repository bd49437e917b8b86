// giant.cuh -- device code shared by the multi-block giant-row kernels (giant.cu) and the persistent
// class steps (sweep.cu).
#pragma once

#include "internal.cuh"

namespace lv {

constexpr int kChunk = 2048;    // arcs per chunk (merge, modularity, compaction)
constexpr int kLmChunk = 512;   // arcs per chunk of the local-moving phase (2 per thread)
constexpr int kSliceLog = 10;   // merge: 1024 table slots (32 bitmap words) per slice
constexpr int kRangeLog = 10;   // local move: 1024 table slots (32 bitmap words) per warp range
constexpr int kLocLog = 12;     // shared pre-aggregation table: 4096 slots >= 2 x kChunk keys

template <class V>
__device__ __forceinline__ V* slot_val(int32_t* kv, unsigned s) {
  return reinterpret_cast<V*>(&kv[2 * (size_t)s + 1]);
}

// tbl_add for a giant's table (kv, at pool offset `base`) that also sets the slot's bit in the
// pool's occupancy bitmap when it claims the slot, so the scan visits only occupied slots.
// Probing starts at slot s (the key's home) whose key was already read as k0.
// An empty slot is claimed together with its first value by one 64-bit compare-and-swap of the
// pair ({kEmpty, 0} -> {key, w}); a slot that holds the key gets an add.
template <class V>
__device__ __forceinline__ bool tbl_add_mark_at(int32_t* kv, unsigned size, int32_t key, V w, unsigned* bits,
                                                int64_t base, unsigned s, int32_t k0) {
  const unsigned long long mine = ((unsigned long long)val_bits<V>(w) << 32) | (uint32_t)key;
  for (unsigned p = 0; p < size; p++) {
    const int32_t k = p == 0 ? k0 : *((volatile int32_t*)&kv[2 * (size_t)s]);
    if (k == key) { atomicAdd(slot_val<V>(kv, s), w); return true; }
    if (k == kEmpty) {
      const unsigned long long old =
          atomicCAS(reinterpret_cast<unsigned long long*>(&kv[2 * (size_t)s]), kEmptyPair, mine);
      if (old == kEmptyPair) {
        atomicOr(&bits[(base + s) >> 5], 1u << ((base + s) & 31));
        return true;
      }
      if ((int32_t)(uint32_t)old == key) { atomicAdd(slot_val<V>(kv, s), w); return true; }
    }
    s = (s + 1) & (size - 1);
  }
  return false;
}

template <class V>
__device__ __forceinline__ bool tbl_add_mark(int32_t* kv, unsigned size, int shift, int32_t key, V w, unsigned* bits,
                                             int64_t base) {
  const unsigned s = tbl_home(key, shift);
  return tbl_add_mark_at(kv, size, key, w, bits, base, s, *((volatile int32_t*)&kv[2 * (size_t)s]));
}

// Where a giant's activity comes from: fast mode snapshots it in k_glm_activate (a neighbour in the
// same random class may re-mark the giant while its step runs); the deterministic mode reads it
// from the flags directly in every kernel of the step -- a colour class is an independent set, so
// nothing marks one of its giants during the step -- and its decide kernel then does what the
// activation did (clears the flag, resets K_i->d, sets the moved mark, counts), one launch fewer.
struct GiantAct {
  int snap = 1;                  // 1: p.active (fast); 0: read below (deterministic)
  int pruning = 0;
  const uint8_t* flags = nullptr;
  const GraphCtl* gc = nullptr;
  const int32_t* vg = nullptr;
};
__device__ __forceinline__ bool giant_active(const GiantAct& ga, const GiantPlan& p, int64_t k, int32_t v) {
  if (ga.snap) return p.active[k] != 0;
  if (ga.gc && *(const volatile int32_t*)&ga.gc[ga.vg[v]].done) return false;
  return !ga.pruning || ga.flags[v] != 0;
}

}  // namespace lv
