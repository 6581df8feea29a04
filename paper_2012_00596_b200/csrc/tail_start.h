// Where a tile of filters (or of the image's filter groups) begins that is as wide as all others and may not go past the end.  Host and
// device code: tests/test_dispatch_cpu.py goes through the tiles of both kernels that use it.
//
// Weights past the last filter are never asked for.  A tensor copy whose box lies past the map's third dimension delivers zeros, but it
// touches the memory that such groups would lie in: the map runs over the whole blob, the fourth dimension's stride is smaller than the
// third's, and the end of the blob may be the end of mapped memory.
#pragma once

#ifdef __CUDACC__
#define NPAS_TAIL_FN __host__ __device__ __forceinline__
#else
#define NPAS_TAIL_FN inline
#endif

namespace npas {

// `width` <= `total`; what the tile has in common with those before it is theirs: its first start - tail_start(...) entries
NPAS_TAIL_FN int tail_start(int start, int width, int total) { return start + width <= total ? start : total - width; }

}  // namespace npas
