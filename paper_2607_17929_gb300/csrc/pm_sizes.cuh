// Mesh sizes, apart from CUDA so that they also compile for the host.
#pragma once

#include <stddef.h>

#include <utility>

namespace pm {

// Every mesh side that a context accepts, 2^a 3^b with a >= 3 up to 1024: what is accepted and what the FFT passes are
// compiled for both come from this list.
constexpr int MESH_SIZES[] = {8,   16,  24,  32,  48,  64,  72,  96,  128, 144, 192,
                              216, 256, 288, 384, 432, 512, 576, 648, 768, 864, 1024};
constexpr size_t NMESHSIZES = sizeof(MESH_SIZES) / sizeof(MESH_SIZES[0]);

constexpr bool is_mesh_size(int n)
{
    for (int m : MESH_SIZES)
        if (m == n) return true;
    return false;
}

// f.template operator()<N>() for the mesh size N = n; false for any other number
template <class F, size_t... I> bool with_mesh_size(int n, F &&f, std::index_sequence<I...>)
{
    return ((n == MESH_SIZES[I] && (f.template operator()<MESH_SIZES[I]>(), true)) || ...);
}
template <class F> bool with_mesh_size(int n, F &&f)
{
    return with_mesh_size(n, f, std::make_index_sequence<NMESHSIZES>{});
}

}  // namespace pm
