// Banded-round kernel instances for at most 8 Krylov directions.
#define FTGCR_THREADS 512
#include "ftgcr_instances.h"
#include "ftgcr_band.cuh"

namespace ftgcr {
const void* band_kernel_k8(bool fp64) {
  return fp64 ? (const void*)k_ftgcr_band<double, 8> : (const void*)k_ftgcr_band<float, 8>;
}
}  // namespace ftgcr
