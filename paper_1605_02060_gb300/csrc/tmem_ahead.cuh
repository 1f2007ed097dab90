// The order in which registers filled by an asynchronous load are named.  Plain C++ apart from the
// execution space, so that the order can be checked on the host with a model of the loads.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define LDDMM_DEVICE __device__ __forceinline__
#else
#define LDDMM_DEVICE inline
#endif

namespace lddmm {

// Chunks of 16 TMEM columns, loaded one ahead of their use.  Ld::issue starts a load into 16
// registers, which hold nothing defined until Ld::wait has returned for those same registers: the
// copy that makes the next chunk the current one therefore comes after the wait that names it, at
// the end of the current chunk's work.
template <typename Ld>
struct TmemAhead {
  uint32_t u[16];     // the current chunk
  uint32_t next[16];  // in flight between ahead() and advance()
  LDDMM_DEVICE void first(uint32_t taddr) {
    Ld::issue(taddr, u);
    Ld::wait(u);
  }
  LDDMM_DEVICE void ahead(uint32_t taddr) { Ld::issue(taddr, next); }
  LDDMM_DEVICE void advance() {
    Ld::wait(next);
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int j = 0; j < 16; ++j) u[j] = next[j];
  }
};

}  // namespace lddmm
