// Sums over the blocks of a co-resident grid, and launches of one cluster, for
// the CG kernels.
//
// One exchange is a reduction and a grid barrier in one: warp 0 of a block
// writes the block's partial, with the exchange's number in the same 16-byte
// store, into every block's inbox, then polls its own inbox and adds the
// values in block order: the total is the same in every block and run. No
// cache line is polled by more than one SM. When every block polled one
// shared array of 152 slots instead (or an atomic counter, or the totals of
// groups of 16), the polls of the waiting blocks held up the stores of the
// late ones: a CG iteration over 147 blocks (32^3 nodes, two exchanges) took
// 14.7 us by one shared array, 16.4 us by a tree of inboxes of 16 (three
// hops), 11.8 us with an atomic counter and 8.4 us by inboxes.
//
// kData: the exchange also orders the blocks' global writes before it ahead
// of the others' reads after it (2,000 of its 7,000 SM cycles). Without it an
// exchange still orders a block's reads before it ahead of the others' writes
// after it where the values read went into the sum.
//
// The inboxes alternate between two sets: a block can be one exchange ahead
// of another, never two. Waits are bounded (4e9 SM cycles, about 2 s): then
// the timeout flag is set and every block returns.
#pragma once

#include <cuda_runtime.h>

namespace pic {

struct alignas(16) GridSlot {
  unsigned long long v, number;
};

__device__ __forceinline__ void slot_put(GridSlot* s, unsigned long long v, unsigned long long number) {
  asm volatile("{ .reg .b128 t; mov.b128 t, {%1, %2}; st.relaxed.gpu.global.b128 [%0], t; }" ::"l"(s), "l"(v),
               "l"(number)
               : "memory");
}
__device__ __forceinline__ void slot_get(const GridSlot* s, unsigned long long& v, unsigned long long& number) {
  asm volatile("{ .reg .b128 t; ld.relaxed.gpu.global.b128 t, [%2]; mov.b128 {%0, %1}, t; }"
               : "=l"(v), "=l"(number)
               : "l"(s)
               : "memory");
}
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

constexpr long long kExchangeCycles = 4000000000LL;
constexpr int kExchangePoll = 5;                           // slots a lane polls
constexpr int kMaxExchangeBlocks = 32 * kExchangePoll;     // 160

// slots of the inboxes of G blocks: two sets of two values
inline constexpr size_t exchange_slots(size_t G) { return 4 * G * G; }

// What a block knows about its launch's exchanges (the same in every thread).
struct GridExchange {
  GridSlot* slots;   // [2 sets][2 values][G inboxes][G]
  int G;             // at most kMaxExchangeBlocks
  unsigned launch;   // unique on these slots, not zero
  unsigned phase;    // exchanges done
  int* timed_out;    // number of a launch that timed out
  int* flags;        // sticky context flags
  int* ok;           // shared: 0 once a wait ran out

  // Totals over the grid of kN (0: a plain barrier, 1 or 2) FP64 values per
  // thread, valid in warp 0. sh: kN blockDim.x doubles of shared memory. The
  // block's values are added by warp 0 alone: a warp's FP64 instruction
  // takes the SM's FP64 pipe for 19 cycles, so a shuffle tree in every warp
  // would cost its warps times as much. The caller follows with a
  // __syncthreads and reads *ok.
  template <int kN, bool kData>
  __device__ __forceinline__ void sum(const double* v, double* tot, double* sh) {
    const int t = threadIdx.x, T = blockDim.x;
    ++phase;
#pragma unroll
    for (int q = 0; q < kN; ++q) sh[q * T + t] = v[q];
    __syncthreads();  // the block's writes before the exchange are done too
    if (t >= 32) return;
    constexpr int kV = kN > 0 ? kN : 1;
    const unsigned long long number = (unsigned long long)launch << 32 | phase;
    GridSlot* set = slots + (size_t)(phase & 1u) * 2 * G * G;
    unsigned long long mine[kV];
#pragma unroll
    for (int q = 0; q < kV; ++q) {
      mine[q] = 0;
      if (kN > 0) {
        double s = sh[q * T + t];
        for (int w = t + 32; w < T; w += 32) s += sh[q * T + w];
        mine[q] = (unsigned long long)__double_as_longlong(warp_sum_d(s));
      }
    }
    // Every publishing lane fences for itself: a release is a fence and the
    // store that follows it in the same thread (lane t's slots are what the
    // blocks t, t + 32, ... read).
    if (kData) fence_gpu();
#pragma unroll
    for (int q = 0; q < kV; ++q)
      for (int i = t; i < G; i += 32) slot_put(set + ((size_t)q * G + i) * G + blockIdx.x, mine[q], number);
    unsigned long long u[kV][kExchangePoll];
    bool good = true;
    const long long t0 = clock64();
    for (int round = 1;; ++round) {
      bool all = true;
#pragma unroll
      for (int q = 0; q < kV; ++q) {
        const GridSlot* inbox = set + ((size_t)q * G + blockIdx.x) * G;
        unsigned long long e[kExchangePoll];
#pragma unroll
        for (int k = 0; k < kExchangePoll; ++k) {
          e[k] = number;
          u[q][k] = 0;
          if (32 * k + t < G) slot_get(inbox + 32 * k + t, u[q][k], e[k]);
        }
#pragma unroll
        for (int k = 0; k < kExchangePoll; ++k) all = all && e[k] == number;
      }
      if (all) break;
      if ((round & 255) == 0 && (clock64() - t0 > kExchangeCycles || *(volatile unsigned*)timed_out == launch)) {
        good = false;
        break;
      }
    }
    good = __all_sync(0xffffffffu, good);
#pragma unroll
    for (int q = 0; q < kN; ++q) {
      double x[kExchangePoll];
#pragma unroll
      for (int k = 0; k < kExchangePoll; ++k) x[k] = __longlong_as_double((long long)u[q][k]);
      static_assert(kExchangePoll == 5, "the tree below adds five values");
      tot[q] = warp_sum_d(((x[0] + x[1]) + (x[2] + x[3])) + x[4]);
    }
    if (kData) fence_gpu();
    if (t == 0) {
      if (!good) {
        atomicExch((unsigned*)timed_out, launch);
        atomicOr(flags, 4);
      }
      *ok = good ? 1 : 0;
    }
  }
};

// A launch of one thread-block cluster.
struct ClusterLaunch {
  cudaLaunchAttribute at = {};
  cudaLaunchConfig_t cfg = {};
  ClusterLaunch(int blocks, int threads, cudaStream_t stream) {
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)blocks;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = stream;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
  }
  ClusterLaunch(const ClusterLaunch&) = delete;

  // Whether the SMs that this process and stream may use hold it. Sixteen
  // blocks need most of a GPC; where a process gets a share of the SMs they may
  // not fit, and the solve takes the grid.
  bool fits(const void* fn) const {
    int n = 0;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, fn, &cfg);
    if (e == cudaSuccess) return n > 0;
    cudaGetLastError();
    return false;
  }
};

}  // namespace pic
