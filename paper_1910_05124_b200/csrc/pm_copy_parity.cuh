// Which phase of its mbarrier a repeated asynchronous copy completes.  Plain C++, so that it can be tested without a GPU.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define PM_DEVICE_INLINE __device__ __forceinline__
#else
#define PM_DEVICE_INLINE inline
#endif

namespace pm {

// A barrier's wait on a parity succeeds when the phase of that parity has completed, so a wait on the parity BEFORE the copy in
// flight succeeds at once.  The parity therefore moves on only with a copy that has been seen to land: after a wait that gave up,
// drain() still polls that copy.
struct CopyParity {
  uint32_t parity = 0;        // of the copy in flight, or of the next one
  // wait(parity): has the copy landed (false: gave up)?
  template <class Wait> PM_DEVICE_INLINE bool await(Wait wait) {
    const bool landed = wait(parity);
    if (landed) parity ^= 1u;
    return landed;
  }
  // polls landed(parity) while more() allows
  template <class Landed, class More> PM_DEVICE_INLINE void drain(Landed landed, More more) const {
    while (!landed(parity) && more()) {}
  }
};

}  // namespace pm
