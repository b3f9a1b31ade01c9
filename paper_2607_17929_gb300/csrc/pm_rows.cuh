// Walks over the particles of a row of cells, apart from the kernels so that they also compile for the host.
#pragma once

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

}  // namespace pm
