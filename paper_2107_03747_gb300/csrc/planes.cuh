// planes.cuh -- the six planes of a site and the clover scratch, shared by the stage kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "lattice.cuh"

namespace tgf {

// Plane index of (mu, nu), mu < nu, in the order 01, 23, 02, 13, 03, 12 (consecutive planes
// pair up in the topological charge); -1 for mu >= nu.
static __constant__ int8_t c_plane_of[4][4] = {{-1, 0, 2, 4}, {-1, -1, 5, 3}, {-1, -1, -1, 1}, {-1, -1, -1, -1}};
// The link direction through which the clover halves of each plane are built (mu of c_clover_owner[mu][nu] = 1): in a
// measured stage 01, 02 by warp 0, 12, 13 by warp 1, 23 by warp 2, 30 by warp 3 -- two planes at most per warp.
// Kernels that build nothing else (mode 2) give c_half's six (mu, nu) to three warps, two each: with a warp per
// direction two of four would have one plane and idle half the time (97 us instead of 83 for 2 x 12x12x36x36 in FP32,
// 256 instead of 224 for 4 x 7x7x21x21 in FP64).
static __constant__ int8_t c_clover_owner[4][4] = {{0, 1, 1, 0}, {0, 0, 1, 1}, {0, 0, 0, 1}, {1, 0, 0, 0}};
static __constant__ int8_t c_half[6][2] = {{0, 1}, {0, 2}, {1, 2}, {1, 3}, {2, 3}, {3, 0}};

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
