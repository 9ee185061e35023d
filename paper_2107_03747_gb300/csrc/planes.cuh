// planes.cuh -- the six planes of a site and the clover scratch, shared by the stage kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "lattice.cuh"

namespace tgf {

// Plane index of (mu, nu), mu < nu, in the order 01, 23, 02, 13, 03, 12 (consecutive planes
// pair up in the topological charge); -1 for mu >= nu.
static __constant__ int8_t c_plane_of[4][4] = {{-1, 0, 2, 4}, {-1, -1, 5, 3}, {-1, -1, -1, 1}, {-1, -1, -1, -1}};
// Which direction's warp builds the clover halves of each plane: 01, 02 by warp 0; 12, 13 by
// warp 1; 23 by warp 2; 03 by warp 3 -- two planes at most per warp instead of 3, 2, 1, 0.
static __constant__ int8_t c_clover_owner[4][4] = {{0, 1, 1, 0}, {0, 0, 1, 1}, {0, 0, 0, 1}, {1, 0, 0, 0}};

// The anti-Hermitian part D - D^+ of a 3x3 matrix as 9 reals (2 Im D_jj; D_jk - conj(D_kj), j<k),
// written to one slot of the clover scratch (AhStore).
template <class T>
__device__ __forceinline__ void store_ah(T* __restrict__ p, int Vp, int s, const mat3<T>& d) {
    const T v[9] = {T(2) * d.e[0][0].im,           T(2) * d.e[1][1].im,           T(2) * d.e[2][2].im,
                    d.e[0][1].re - d.e[1][0].re, d.e[0][1].im + d.e[1][0].im, d.e[0][2].re - d.e[2][0].re,
                    d.e[0][2].im + d.e[2][0].im, d.e[1][2].re - d.e[2][1].re, d.e[1][2].im + d.e[2][1].im};
    AhStore<T>::store(p, Vp, s, v);
}

}  // namespace tgf
