// Bookkeeping of asynchronous loads into a ring of two buffers (compiled for the host too, where its test runs).
#pragma once

#ifdef __CUDACC__
#define JAB_BOXES_FN __host__ __device__ __forceinline__
#else
#define JAB_BOXES_FN inline
#endif

namespace jab {

// Load n goes to buffer n & 1, whose barrier completes phase n >> 1 with it. `wait(buffer, parity)` is a bounded
// wait for that phase. A wait that gave up leaves its load in flight: it is not counted as landed, so that
// drain() waits for it, and for the one behind it, before the shared memory goes to another block.
struct TwoBoxes {
  int issued = 0, landed = 0;
  JAB_BOXES_FN int next() const { return issued & 1; }  // buffer of the load to issue
  template <class Wait>
  JAB_BOXES_FN bool take(Wait wait) {
    if (!wait(landed & 1, (unsigned)(landed >> 1) & 1u)) return false;
    ++landed;
    return true;
  }
  template <class Wait>
  JAB_BOXES_FN void drain(Wait wait) {
    for (; landed < issued; ++landed) wait(landed & 1, (unsigned)(landed >> 1) & 1u);
  }
};

}  // namespace jab
