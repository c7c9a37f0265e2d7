// Halo exchange between the y-slabs of one grid on one device.
#pragma once

#include "kbc_kernels.cuh"

namespace kbc {

constexpr int kSlabFaces = 32;  // faces per launch (1 KB of kernel parameters)

// One face: three population rows of one slab's boundary, pitch bytes apart,
// into a ghost row of its neighbour.
struct SlabFace {
    const char* src;
    char* dst;
    long long src_pitch, dst_pitch;
};
struct SlabFaces {
    SlabFace face[kSlabFaces];
};

// blockIdx.y: the face; units of U per row.  Moves a few hundred KB a step,
// so its time is a launch's; what it replaces is four copies per slab through
// staging buffers.
template <class U>
__global__ void __launch_bounds__(256) slab_halos(SlabFaces f, int units)
{
    chain_enter();
    const SlabFace& s = f.face[blockIdx.y];
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < 3 * units; q += gridDim.x * blockDim.x) {
        const int p = q / units, c = q - p * units;
        reinterpret_cast<U*>(s.dst + p * s.dst_pitch)[c] =
            ld_field(reinterpret_cast<const U*>(s.src + p * s.src_pitch) + c);
    }
}

}  // namespace kbc
