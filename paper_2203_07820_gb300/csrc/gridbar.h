// Bounded grid-wide barrier of the cooperative kernels (all CTAs co-resident).
#pragma once

#include <cuda_runtime.h>

#include "../../include/dftfe_gb300.h"

namespace dftfe {
namespace jac {

constexpr long kBarrierSpins = 20000000L;   // x 64 ns sleep: about a second

struct Barrier {
  unsigned int count;
  unsigned int gen;
  int abort;
  unsigned int reads;   // CTAs that have read the rotation inputs, summed over rounds
  long long limit;      // spin iterations before a wait gives up
  unsigned int missing; // arrivals the barrier expects beyond the grid (0; 1 only in the wait test)
  unsigned long long top;   // bits of the largest |entry| of the matrix (k_tridiag)
};

// every call starts from a cleared barrier with its spin limit and expected arrivals (dense.cu)
void init_barrier(cudaStream_t s, Barrier* b, long long limit, unsigned int missing);

#ifdef __CUDACC__
// grid-wide barrier (all CTAs are co-resident under the cooperative launch); false when
// a wait ran out or another CTA gave up
__device__ __forceinline__ bool grid_barrier(Barrier* b, int* status) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    ok = 1;
    volatile unsigned int* vgen = &b->gen;
    volatile int* vabort = &b->abort;
    const unsigned int g = *vgen;
    const long long lim = b->limit;
    __threadfence();
    if (atomicAdd(&b->count, 1u) == gridDim.x - 1 + b->missing) {
      atomicExch(&b->count, 0u);
      __threadfence();
      atomicAdd(&b->gen, 1u);
    } else {
      long long it = 0;
      while (*vgen == g) {
        if (*vabort || ++it > lim) {
          ok = 0;
          atomicExch(&b->abort, 1);
          atomicCAS(status, 0, (int)DFTFE_ERR_TIMEOUT);
          break;
        }
        __nanosleep(64);
      }
    }
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}
#endif  // __CUDACC__

}  // namespace jac
}  // namespace dftfe
