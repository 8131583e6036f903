// The span [lo, hi] of 64-bit keys that the select of the Gamma builder narrows, bin by bin.  Keys may lie anywhere in 64 bits: a score that is
// a NaN with its sign set is a key just below 2^64, so that no step may pass the end of the span it starts from.  Plain arithmetic: the host
// compiler takes it, too.
#pragma once

#ifdef __CUDACC__
#define BSP_SPAN_FN __host__ __device__ __forceinline__
#else
#define BSP_SPAN_FN inline
#endif

namespace bsp {

// log2 of the width of a bin: the span lo < hi falls into at most 2^width of them.
BSP_SPAN_FN int span_shift(unsigned long long lo, unsigned long long hi, int width)
{
#ifdef __CUDA_ARCH__
    const int bits = 64 - __clzll((long long)(hi - lo));
#else
    const int bits = 64 - __builtin_clzll(hi - lo);
#endif
    return bits > width ? bits - width : 0;
}

// The part of the span that bin `bin` covers.
BSP_SPAN_FN void span_to_bin(unsigned long long &lo, unsigned long long &hi, unsigned bin, int shift)
{
    lo += (unsigned long long)bin << shift;
    const unsigned long long rest = (1ull << shift) - 1ull;
    if (hi - lo > rest) hi = lo + rest;
}

// Rounds after which every span is one key: a round leaves at most 2^shift of what were 2^(shift + width).
BSP_SPAN_FN constexpr int span_rounds(int width) { return (64 + width - 1) / width; }

}  // namespace bsp
