// pack.cu -- canonical FP64 link layout <-> device storage planes.
//
// Canonical: per configuration [site][mu][row][col][re,im] doubles (x0 fastest within site).
// For these launches CfgDesc::x_off is the configuration's offset in the canonical buffer
// (doubles) and blocks cover 32 sites x 4 directions (one thread per link).
#include <cuda_runtime.h>

#include "lattice.cuh"

namespace tgf {

// Both kernels are bound by HBM: a site takes 576 canonical bytes and 192-576 stored ones.  The canonical field is read
// and written in its own order, consecutive threads on consecutive doubles, and the links change hands in
// shared memory, a site per row of 73 (odd: the rows of a warp's lanes start in different banks).  A thread that
// moved its link's 18 doubles itself touched 32 sectors per store, 8 bytes of each: 4 x 16x16x48x48 in FP32
// packed in 403 us and unpacked in 1185 us (2.04 GB each, 306 us at 6.67 TB/s); now 283 and 311.
constexpr int kRow = 73;

// float -> double.  The FP64 pipe converts 1.9 lanes per clock and SM (294 us for the 170 million entries of
// that field); a normal number widens by three shifts of its bits, which the integer pipe has to spare.
__device__ __forceinline__ double widen(float x) {
    const unsigned u = __float_as_uint(x);
    if (((u + 0x00800000u) & 0x7f000000u) == 0) return (double)x;  // 0, subnormal, infinite or NaN
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))), (int)(u << 29));
}
__device__ __forceinline__ double widen(double x) { return x; }

template <int P, int CAP>
__global__ void __launch_bounds__(128)
k_pack(const __grid_constant__ BatchT<CAP> B, const double* __restrict__ canon, typename Store<P>::T* __restrict__ w) {
    using T = typename Store<P>::T;
    __shared__ T buf[32 * kRow];
    const int ci = find_cfg(B, blockIdx.x);
    const CfgDesc& c = B.c[ci];
    const int s0 = (blockIdx.x - c.blk0) * 32, mu = threadIdx.x >> 5, lane = threadIdx.x & 31, s = s0 + lane;
    const double* src = canon + c.x_off + (size_t)s0 * 72;
    const int n = min(32, c.V - s0) * 72;
#pragma unroll
    for (int k = 0; k < 18; ++k) {
        const int i = k * 128 + threadIdx.x;
        if (i < n) buf[i + i / 72] = (T)__ldg(src + i);
    }
    __syncthreads();
    if (s >= c.V) return;
    mat3<T> u;
    const T* row = buf + lane * kRow + mu * 18;
#pragma unroll
    for (int k = 0; k < 9; ++k) u.e[k / 3][k % 3] = {row[2 * k], row[2 * k + 1]};
    Store<P>::store(w + c.w_off + (size_t)mu * Store<P>::reals * c.Vp, c.Vp, s, u);
}

template <int P, int CAP>
__global__ void __launch_bounds__(128)
k_unpack(const __grid_constant__ BatchT<CAP> B, const typename Store<P>::T* __restrict__ w, double* __restrict__ canon) {
    using T = typename Store<P>::T;
    __shared__ T buf[32 * kRow];
    const int ci = find_cfg(B, blockIdx.x);
    const CfgDesc& c = B.c[ci];
    const int s0 = (blockIdx.x - c.blk0) * 32, mu = threadIdx.x >> 5, lane = threadIdx.x & 31, s = s0 + lane;
    if (s < c.V) {
        mat3<T> u;
        Store<P>::load(w + c.w_off + (size_t)mu * Store<P>::reals * c.Vp, c.Vp, s, u);
        T* row = buf + lane * kRow + mu * 18;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            row[2 * k] = u.e[k / 3][k % 3].re;
            row[2 * k + 1] = u.e[k / 3][k % 3].im;
        }
    }
    __syncthreads();
    double* dst = canon + c.x_off + (size_t)s0 * 72;
    const int n = min(32, c.V - s0) * 72;
#pragma unroll
    for (int k = 0; k < 18; ++k) {
        const int i = k * 128 + threadIdx.x;
        if (i < n) dst[i] = widen(buf[i + i / 72]);
    }
}

template <int P>
static void pack_p(const Batch& B, const double* canon, void* w, cudaStream_t st) {
    using T = typename Store<P>::T;
    if (B.ncfg <= kSmallCap) {
        BatchT<kSmallCap> b;
        b.ncfg = B.ncfg;
        b.nblk = B.nblk;
        for (int i = 0; i < B.ncfg; ++i) b.c[i] = B.c[i];
        k_pack<P, kSmallCap><<<B.nblk, 128, 0, st>>>(b, canon, (T*)w);
    } else {
        k_pack<P, kMaxCfg><<<B.nblk, 128, 0, st>>>(B, canon, (T*)w);
    }
}

template <int P>
static void unpack_p(const Batch& B, const void* w, double* canon, cudaStream_t st) {
    using T = typename Store<P>::T;
    if (B.ncfg <= kSmallCap) {
        BatchT<kSmallCap> b;
        b.ncfg = B.ncfg;
        b.nblk = B.nblk;
        for (int i = 0; i < B.ncfg; ++i) b.c[i] = B.c[i];
        k_unpack<P, kSmallCap><<<B.nblk, 128, 0, st>>>(b, (const T*)w, canon);
    } else {
        k_unpack<P, kMaxCfg><<<B.nblk, 128, 0, st>>>(B, (const T*)w, canon);
    }
}

void launch_pack(int prec, const Batch& B, const double* canon, void* w, cudaStream_t st) {
    if (prec == P64) pack_p<P64>(B, canon, w, st);
    else if (prec == P32) pack_p<P32>(B, canon, w, st);
    else pack_p<P32R12>(B, canon, w, st);
}

void launch_unpack(int prec, const Batch& B, const void* w, double* canon, cudaStream_t st) {
    if (prec == P64) unpack_p<P64>(B, w, canon, st);
    else if (prec == P32) unpack_p<P32>(B, w, canon, st);
    else unpack_p<P32R12>(B, w, canon, st);
}

TGF_CHECK_WORD(pack)

}  // namespace tgf
