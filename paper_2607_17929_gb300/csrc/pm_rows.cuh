// Walks over the particles of a row of cells, apart from the kernels so that they also compile for the host.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define PM_HD __host__ __device__ __forceinline__
#else
#define PM_HD inline
#endif

namespace pm {

// f(c) for c = 0, 32, 64, .. below n.  A context takes up to 2^31 - 1 particles, and all of them may lie in one row:
// from n = 2^31 - 31 on the count past the last group does not fit an int.  c + 31 does.
template <class F> PM_HD void for_groups(int n, F &&f)
{
    for (unsigned c = 0; c < (unsigned)n; c += 32) f((int)c);
}

// Tiles of k_mass: 9^3 cells, staged MCAP particles at a time.
constexpr int MCAP = 960;   // (a nearly uniform load of one per cell has 729)

// Whether a tile's particle count, or the count at the end of its last chunk, may pass 2^31 - 1, so that its offsets
// need 64 bits.  The tile of an 8^3 mesh reaches round the box: it holds the cells of its far faces twice along each
// axis, a corner cell eight times.
PM_HD bool mass_wide(int n, int64_t np) { return (n == 8 ? 8 * np : np) > (int64_t)INT32_MAX - MCAP; }

}  // namespace pm
