// Bookkeeping of an operand ring: slots 0 .. stages - 1 filled in turn, round after round, each with a barrier whose
// phase flips when the slot's copies have landed.
#pragma once

#ifdef __CUDACC__
#define XL_HD __host__ __device__ __forceinline__
#else
#define XL_HD inline
#endif

namespace xl {

// Parity of the phase of slot s's last use, -1 when it has not been used: `slot` is the next one to be filled,
// `ph` the parity of its round and `first` says that this is the ring's first round.
XL_HD int ring_last_use(unsigned slot, unsigned ph, bool first, unsigned s) {
  return s < slot ? (int)ph : first ? -1 : (int)(ph ^ 1u);
}

}  // namespace xl
