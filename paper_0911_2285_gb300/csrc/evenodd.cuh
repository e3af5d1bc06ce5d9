// Half-lattice indexing of the even-odd operator (evenodd.cu, reliable.cu).
#pragma once
#include "common.cuh"

namespace lqcd {

// Full site index of half index h in parity P.
__device__ __forceinline__ int eo_site(const Geom& g, int h, int P) {
    const int s0 = 2 * h;
    int r = s0 / g.L[0];
    const int y = r % g.L[1];
    r /= g.L[1];
    const int z = r % g.L[2], t = r / g.L[2];
    // x of s0 is even, so the parity of s0 is that of y + z + t
    return s0 + ((((y + z + t) & 1) != P) ? 1 : 0);
}

// A half field read at full site indices (the neighbours of a site of the other parity).
template <typename S> struct HalfIn {
    const void* p;
    int Vh;
    template <typename C> __device__ __forceinline__ void load(int s, C (&v)[12]) const {
        Field<S>::load(p, Vh, s >> 1, v);
    }
};

}  // namespace lqcd
