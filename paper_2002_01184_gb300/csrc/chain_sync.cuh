// How the CTAs of an adapting multi-transition launch meet (elementwise_chain.cu,
// logreg_chain.cu).
//
// A statistic -- an acceptance probability or a sum of eight, never negative --
// reaches the other CTAs in one 64-bit word whose sign bit says whether it has
// been written: a transition uses one of two sets of slots, and each use of a
// slot flips the sign that means "written".  The word that announces the value
// is the value, so no fence, arrival counter or second read lies between the
// last CTA's store and everyone's sum.  A slot is reused two transitions later:
// a CTA that writes it has seen every CTA's next statistic, so all have read it.
// Between launches every slot holds kEmptySlot.
#pragma once
#include "hmc_device.cuh"
#include "hmc_internal.h"
#include "sm100_ptx.cuh"

namespace hmc {

constexpr unsigned long long kEmptySlot = ~0ull;
constexpr unsigned long long kSlotSign = 1ull << 63;

__device__ __forceinline__ void put_slot(unsigned long long* p, double v, bool negative) {
  const unsigned long long w = static_cast<unsigned long long>(__double_as_longlong(v)) | (negative ? kSlotSign : 0ull);
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}

__device__ __forceinline__ unsigned long long read_slot(const unsigned long long* p) {
  unsigned long long w;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
  return w;
}

__device__ __forceinline__ double slot_value(unsigned long long w) {
  return __longlong_as_double(static_cast<long long>(w & ~kSlotSign));
}

// The adaptation state's next update from the sum over C chains, with
// inv_c = 1 / n_c rounded: the mean is correctly rounded (Markstein 1990: the
// rounded reciprocal's quotient, corrected by its exact remainder).
__device__ __forceinline__ void da_apply_sum(DAState* s, const DACoef& c, double sum, double n_c, double inv_c,
                                             long long t) {
  const double q = sum * inv_c;
  da_apply(s, c, fma(fma(-q, n_c, sum), inv_c, q), t);
}

// Leaving an adapting launch (all threads): CTA 0 writes the adaptation state
// (every CTA has read it: all have passed a meeting), and the last CTA out
// empties `n` slots for the next launch.
__device__ __forceinline__ void leave_adapting(DAState* da, DAState* mine, unsigned* left, unsigned long long* slots,
                                               int64_t n) {
  __shared__ int last_s;
  if (threadIdx.x == 0) {
    if (blockIdx.x == 0) {
      mine->arrive = 0u;
      *da = *mine;
    }
    __threadfence();
    last_s = atomicAdd(left, 1u) == gridDim.x - 1u ? 1 : 0;
  }
  __syncthreads();
  if (last_s) {
    for (int64_t b = threadIdx.x; b < n; b += blockDim.x) slots[b] = kEmptySlot;
    if (threadIdx.x == 0) *left = 0u;
  }
}

}  // namespace hmc
