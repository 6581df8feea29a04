// The ranges of keys that the layer-wide selection of prune.cu narrows down, one pass after the other.  Host and device code, so that its
// ends can be checked on keys up to 2^64 - 1 without a GPU (tests/test_select_range_cpu.py).
//
// A key is the bit pattern of a sum of squares, which is never negative; but a sum that is no number keeps its sign and payload, so any
// 64-bit pattern may come.  The first pass lays kSelBins bins over what lies between two sampled keys, with an open bin at either end;
// every later one over the range [lo, hi] that the pass before picked.  A picked bin holds a key, so its first key lies inside the range
// divided, and its last one is found from there without leaving it.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define NPAS_SEL_FN __host__ __device__ __forceinline__
#else
#define NPAS_SEL_FN inline
#endif

namespace npas {

constexpr unsigned kSelBins = 1024;
// A first pass may leave 64 bits of range; each later one leaves ten less: 54, 44, 34, 24, 14, 4 and a single value.
constexpr int kSelPasses = 8;

NPAS_SEL_FN int sel_bits(uint64_t v)
{
#ifdef __CUDA_ARCH__
    return v ? 64 - __clzll((long long)v) : 0;
#else
    return v ? 64 - __builtin_clzll(v) : 0;
#endif
}
NPAS_SEL_FN int sel_shift(uint64_t span) { return sel_bits(span) > 10 ? sel_bits(span) - 10 : 0; }

// first pass: bins of 2^shift keys from `base` on, one below and the last one open
NPAS_SEL_FN int sel_first_shift(uint64_t base, uint64_t top)
{
    const int shift = sel_shift(top - base);
    return (top - base) >> shift > kSelBins - 3 ? shift + 1 : shift;
}
NPAS_SEL_FN unsigned sel_first_bin(uint64_t k, uint64_t base, int shift)
{
    const uint64_t b = (k - base) >> shift;
    return k < base ? 0u : b < kSelBins - 2 ? 1u + (unsigned)b : kSelBins - 1;
}
// the last of the 2^shift keys from `lo` on, or `most`, which is not below `lo`  (lo + 2^shift may lie past 2^64)
NPAS_SEL_FN uint64_t sel_last(uint64_t lo, int shift, uint64_t most)
{
    const uint64_t span = (1ull << shift) - 1;
    return most - lo > span ? lo + span : most;
}
NPAS_SEL_FN void sel_first_range(unsigned bin, uint64_t base, int shift, uint64_t &lo, uint64_t &hi)
{
    lo = bin == 0 ? 0 : base + ((uint64_t)(bin - 1) << shift);
    hi = bin == 0 ? base - 1 : bin == kSelBins - 1 ? ~0ull : sel_last(lo, shift, ~0ull);
}

// later passes: bins of 2^shift keys from `lo` on
NPAS_SEL_FN unsigned sel_bin(uint64_t k, uint64_t lo, int shift) { return (unsigned)((k - lo) >> shift); }
NPAS_SEL_FN void sel_range(unsigned bin, int shift, uint64_t &lo, uint64_t &hi)
{
    lo += (uint64_t)bin << shift;
    hi = sel_last(lo, shift, hi);
}

}  // namespace npas
