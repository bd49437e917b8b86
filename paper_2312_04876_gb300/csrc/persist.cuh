// persist.cuh -- barriers of the persistent kernels (colouring rounds, narrow class steps).
//
// A persistent kernel runs many dependent steps in one launch.  What a step costs beyond its work is
// the barrier between steps, so the launch takes the smallest scope that holds a step's work:
//   kCta      one block: __syncthreads, tens of nanoseconds;
//   kCluster  one thread-block cluster: the hardware cluster barrier, a few hundred nanoseconds;
//   kGrid     one block per SM, launched cooperatively: an arrival counter in L2, about two
//             microseconds.
// Only the grid barrier can wait on something that is not scheduled, so it is bounded: a block that
// polls longer than max_spins sets kErrTimeout and leaves, the others see the bit and leave too.
#pragma once

#include "internal.cuh"

namespace lv {

enum Scope { kCta = 0, kCluster = 1, kGrid = 2 };

constexpr int kClusterBlocks = 8;  // the portable maximum
constexpr long long kBarrierPolls = 1LL << 23;  // built-in bound: x ~0.6 us a poll, about 5 s (a wide step
                                                // of a graph of billions of arcs takes a good part of one)

// Barrier word of one step: arrivals in the high bits, below them a sum the blocks publish with
// their arrival, so that what every block must know about the step (how much work it left) comes
// with the barrier and costs no read after it.
constexpr int kBarShift = 52;
constexpr unsigned long long kBarSum = (1ULL << kBarShift) - 1;

struct PersistBar {
  unsigned long long* word;  // [3] rotating words, zeroed before the launch
  long long max_spins;
  unsigned epoch;            // barriers passed (each block's own copy)
  unsigned from;             // the first barrier max_spins bounds; kBarrierPolls bounds those before (0 but in tests)
};

// Every thread of every block calls it; thread 0 evaluates `value()` (below 2^52 in total) once the
// whole block has arrived, and every thread runs `meanwhile()` between the arrival and the wait (loads
// for the next step that no block of this one writes).  Writes before it are visible after it to all
// blocks of the scope.  *sum = the blocks' values.  Returns false (for the whole block) once a wait has
// run out; the block then leaves.  (The scope is a template argument: as a launch argument it cost a
// one-block round 0.5 us.)
template <int SC, class V, class W>
__device__ __forceinline__ bool scope_barrier(PersistBar& b, Ctrl* ctrl, unsigned long long* sum, V value,
                                              W meanwhile) {
  __shared__ unsigned long long sum_s;
  __syncthreads();
  if constexpr (SC == kCta) {
    if (threadIdx.x == 0) sum_s = value();
    meanwhile();
    __syncthreads();
    *sum = sum_s;
    return true;
  } else {
    // barrier e counts in word e % 3 and clears the next one, last read before barrier e - 1
    unsigned long long* w = b.word + b.epoch % 3;
    unsigned long long* clear = b.word + (b.epoch + 1) % 3;
    b.epoch++;
    if constexpr (SC == kCluster) {
      if (threadIdx.x == 0) {
        const unsigned long long add = value();
        if (add) atomicAdd(w, add);
        if (blockIdx.x == 0) *(volatile unsigned long long*)clear = 0;
      }
      __syncwarp();
      asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
      meanwhile();
      __syncwarp();
      asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
      *sum = *(volatile unsigned long long*)w;
      return true;
    } else {
      __shared__ int ok_s;
      unsigned long long x = 0;
      if (threadIdx.x == 0) {
        if (blockIdx.x == 0) *(volatile unsigned long long*)clear = 0;
        const unsigned long long add = (1ULL << kBarShift) + value();
        asm volatile("atom.add.release.gpu.global.u64 %0, [%1], %2;" : "=l"(x) : "l"(w), "l"(add) : "memory");
        x += add;
      }
      meanwhile();
      if (threadIdx.x == 0) {
        int ok = 1;
        long long spins = 0;
        while ((x >> kBarShift) < gridDim.x) {
          if (++spins > b.max_spins && (b.epoch > b.from || spins > kBarrierPolls)) {
            atomicOr(&ctrl->error, kErrTimeout);
            ok = 0;
            break;
          }
          if ((spins & 63) == 0 && (*(volatile int32_t*)&ctrl->error & kErrTimeout)) {
            ok = 0;
            break;
          }
          asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(x) : "l"(w) : "memory");
        }
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
        sum_s = x & kBarSum;
        ok_s = ok;
      }
      __syncthreads();
      *sum = sum_s;
      return ok_s != 0;
    }
  }
}

template <int SC, class V>
__device__ __forceinline__ bool scope_barrier(PersistBar& b, Ctrl* ctrl, unsigned long long* sum, V value) {
  return scope_barrier<SC>(b, ctrl, sum, value, []() {});
}

// Launches kernel(args) with the scope's grid.  Returns the launch's status: a cluster or a cooperative
// grid may be refused (a context that has only a part of the SMs); one block never is.
template <class... P>
inline cudaError_t scope_launch(Scope sc, const Ctx& c, void (*kernel)(P...), int threads, size_t smem, P... args) {
  if (c.one_block && sc != kCta) return cudaErrorCooperativeLaunchTooLarge;
  if (smem > 48 * 1024) {  // the opt-in is idempotent and costs about a microsecond
    const cudaError_t e = cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(sc == kCta ? 1 : (sc == kCluster ? kClusterBlocks : c.num_sms));
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = c.s;
  cudaLaunchAttribute at[1] = {};
  if (sc == kCluster) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kClusterBlocks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  } else {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
  }
  cfg.attrs = at;
  cfg.numAttrs = sc == kCta ? 0 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace lv
