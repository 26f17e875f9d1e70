// Index arithmetic of a context's rows: up to 2^31 - 1 of them (f2gpu.h), so a
// sum with a step or a chunk beyond the last row does not fit 32 bits.  Plain
// C++, so that a host compiler can check it at the limit.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define F2_HD __host__ __device__ __forceinline__
#else
#define F2_HD inline
#endif

namespace f2 {

// Chunk k of `chunk` items from `from` on, of n: whether there is one.
F2_HD bool chunk_exists(int from, int k, int chunk, int n) { return from + (int64_t)k * chunk < n; }

// The item after a step (or a chunk) from `at` <= n.
F2_HD int step_to(int at, int step, int n) { return n - at < step ? n : at + step; }

// Chunks of the items from..n-1.
F2_HD int chunk_count(int from, int chunk, int n) { return (int)(((int64_t)n - from + chunk - 1) / chunk); }

// Item at + j (at <= n, 0 <= j < 2^31) is one of the n: as a sum of unsigned numbers.
F2_HD bool item_in(int at, int j, int n) { return (uint32_t)at + (uint32_t)j < (uint32_t)n; }

// What rep_count holds for a context whose R > 0 rows all stand for themselves
// (0 .. 2^31 - 1: the number of its representatives, -1: nothing to do).
F2_HD int32_t all_rows(int64_t R) { return (int32_t)(-R - 1); }
F2_HD int rows_of(int32_t count) { return -(count + 1); }

// Entries of a hash table for n rows, a power of two in 64 .. most.
F2_HD int table_entries(int n, int most)
{
    int e = 64;
    while (e < most && e / 2 < n) e <<= 1;
    return e;
}

}  // namespace f2
