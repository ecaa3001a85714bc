// arc_index.h -- arcs of a row at the end of the largest graphs.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define FSGP_HD __host__ __device__ __forceinline__
#else
#define FSGP_HD inline
#endif

namespace fsgp {

// Arc positions are below 2^31, but a loop over a row's arcs steps past the row's end by up to
// its stride: the loops count without sign, or in 64 bits, so that the last rows of the largest
// graphs end.
// arc_in: is arc b + k one of a row that ends at e?
FSGP_HD bool arc_in(int32_t b, int32_t k, int32_t e) { return (uint32_t)b + (uint32_t)k < (uint32_t)e; }

// Chunks of `chunk` arcs that d arcs take.
FSGP_HD int64_t arc_chunks(int32_t d, int32_t chunk) { return ((int64_t)d + chunk - 1) / chunk; }

}  // namespace fsgp
