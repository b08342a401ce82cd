// grid_index.h -- the thread's index in a one-dimensional grid and the row it works on
// when 2^SHIFT threads share one.  64 bits: 32 threads to a row pass 2^32 at 2^27
// rows, and a caller's matrix of few blocks a row can have up to 2^29.
#pragma once

#ifdef __CUDACC__
#define BD_GRID_FN __host__ __device__ __forceinline__
#else
#define BD_GRID_FN inline
#endif

namespace bd {

BD_GRID_FN long long grid_index(unsigned block, unsigned dim, unsigned thread) { return (long long)block * dim + thread; }

template <int SHIFT> BD_GRID_FN int grid_row(unsigned block, unsigned dim, unsigned thread)
{
    return (int)(grid_index(block, dim, thread) >> SHIFT);
}

}  // namespace bd
