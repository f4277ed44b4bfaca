// Index arithmetic shared by kernels, where its range is not obvious. Compiles for the host
// as well (tests/test_index.py).
#pragma once

#include <cuda_runtime.h>

namespace dsrg {

// Element r of an array [nA nA][nV][nV]: xu nV^2 + e nV + f. A 64-bit division is some 40
// instructions for the 16 bytes that an element moves, so the position (e, f) is taken
// apart in 32 bits where nV^2 fits.
__host__ __device__ __forceinline__ void split_xu_ef(size_t r, int nV, int& xu, int& e, int& f) {
  const size_t nV2 = (size_t)nV * nV, q = r / nV2;
  xu = (int)q;
  if (nV <= 65535) {
    const unsigned ef = (unsigned)(r - q * nV2);
    e = (int)(ef / (unsigned)nV);
    f = (int)(ef % (unsigned)nV);
  } else {
    const size_t ef = r - q * nV2;
    e = (int)(ef / nV);
    f = (int)(ef - (size_t)e * nV);
  }
}

}  // namespace dsrg
