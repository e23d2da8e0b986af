// plane.cuh -- access to one plane of a lattice's buffers.
#pragma once

namespace lbm39 {

// Element `index` of a plane, index in [0, 2^31 - 64).  The index is 32-bit and unsigned, and the
// plane's address the same for all threads, so that an address is one multiply-add on a uniform
// base; the byte offset is 64-bit, as a plane of 2^29 doubles has 2^32 bytes.
template <class P>
__device__ __forceinline__ P& at(P* plane, int index) {
  return plane[(unsigned)index];
}

}  // namespace lbm39
