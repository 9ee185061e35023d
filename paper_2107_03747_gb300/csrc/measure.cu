// measure.cu -- observables E, Q, P of every configuration from the clover halves.
//
// The stage kernel (modes 1 and 2) leaves, per site and plane, the two halves of the clover's
// anti-Hermitian part A = C - C^+ (so G = -(i/8) A, eq. gmunu) and the twisted plaquette
// trace.  k_clover_sum adds the halves and accumulates per site
//   e(n) = sum_{mu<nu} |A_{mu nu}|_F^2            (Tr G^2 = |A|^2 / 64)
//   q(n) = <A01,A23> - <A02,A13> + <A03,A12>       (Tr G_a G_b = <A_a,A_b> / 64, <X,Y> = Re sum X conj(Y))
//   s(n) = sum_{mu<nu} (3 - Re Tr[Z* P_{mu nu}(n)])
// in the working precision (the stage kernel stores each plane's 3 - Re Tr[Z* P], so the small
// deviations are summed, not six numbers near 3), then reduces them over the block in FP64 (warp
// shuffles, fixed order) to one partial per block.  The partials of a configuration are summed in a fixed
// order, by its last block or by k_reduce, into {t, E, Q, P, S} with E = sum e/(64 V), Q = sum q/(256 pi^2) (eq. qlatt
// with Gt_{mu nu} = eps_{mu nu rho sigma} G_{rho sigma}/2), S = sum s, P = 1 - S/(18 V).
// Both orders are fixed: results are bitwise reproducible.
#include <cuda_runtime.h>

#include "lattice.cuh"

namespace tgf {

// First observable slot (o_off + 1) whose record came out non-finite since the host last read
// the word; 0 if none.  Read and cleared by nonfinite_read_and_clear().
__device__ unsigned long long g_nonfinite;

unsigned long long nonfinite_read_and_clear(cudaStream_t st, cudaError_t* err) {
    unsigned long long v = 0, z = 0;
    cudaError_t e = cudaMemcpyFromSymbolAsync(&v, g_nonfinite, sizeof v, 0, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyToSymbolAsync(g_nonfinite, &z, sizeof z, 0, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    *err = e;
    return e == cudaSuccess ? v : 0;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

constexpr double kSliceUnit = 1.0 / (256.0 * 3.14159265358979323846 * 3.14159265358979323846);

// Sums of a configuration's partials -> its record {t, E, Q, P, S}.
__device__ __forceinline__ void write_record(const CfgDesc& c, double e, double q, double S, double* __restrict__ obs) {
    const double V = (double)c.V;
    const double pi = 3.14159265358979323846;
    double* o = obs + (size_t)c.o_off * 5;
    const double E = e / (64.0 * V), Q = q / (256.0 * pi * pi);
    o[0] = c.h;                                   // t
    o[1] = E;
    o[2] = Q;
    o[3] = 1.0 - S / (18.0 * V);                  // P = (1/(18V)) sum Re Tr[Z* P]
    o[4] = S;                                     // S = sum (3 - Re Tr[Z* P])
    // a non-finite record (non-finite links in, or an overflow) is reported to the host
    if (!isfinite(E) || !isfinite(Q) || !isfinite(S))
        atomicCAS(&g_nonfinite, 0ull, (unsigned long long)c.o_off + 1ull);
}
// One of the three sums (k = 0, 1, 2: e, q, s) over nb partials, by a warp, in a fixed order.  A configuration's partials
// are summed in four such parts, by whichever kernel does it: the record is the same to the bit.
__device__ __forceinline__ double sum_partials(const double* __restrict__ partial, int nb, int k, int lane) {
    const double* o = partial + k;
    double v0 = 0, v1 = 0;
    int i = lane;
    for (; i + 32 < nb; i += 64) {
        v0 += __ldcg(o + (size_t)i * kPartials);
        v1 += __ldcg(o + (size_t)(i + 32) * kPartials);
    }
    if (i < nb) v0 += __ldcg(o + (size_t)i * kPartials);
    return warp_sum(v0 + v1);
}

// One thread per site, bound by HBM where the lattice is large (4 x 16x16x48x48 in FP32: 1.08 GB in 183 us).  LAST: the last
// block of a configuration to finish (its counter, cleared by the stage kernel that wrote the halves) sums the
// partials, instead of a launch of its own for a few numbers (k_reduce).  That is for launches of few blocks, whose
// time is latency: the 18-step flow of 4x4x12x12, 18 blocks, 295 -> 283 us; with many blocks the fence and the counter
// cost more than the launch (a 6-step flow of 4 x 16x16x48x48 17.10 -> 17.15 ms).  Three threads per site, one for
// each pair of planes, were no faster on the small lattice and 22 % slower on the large one.
template <class T, int CAP, bool LAST>
__global__ void __launch_bounds__(kMeasureSites)
k_clover_sum(const __grid_constant__ BatchT<CAP> B, const T* __restrict__ clov, double* partial, double* __restrict__ obs,
             int traceless) {
    __shared__ double red[kMeasureSites / 32][3];
    __shared__ bool last;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ci = find_cfg(B, blockIdx.x);
    const CfgDesc& c = B.c[ci];
    const int s = (blockIdx.x - c.blk0) * kMeasureSites + threadIdx.x;
    double e = 0, q = 0, pl = 0;
    if (s < c.V) {
        const T* cb = clov + c.m_off;
        const size_t Vp = (size_t)c.Vp;
        T te = T(0), tq = T(0), tp = T(0);
        T a0[9];
#pragma unroll
        for (int p = 0; p < 6; ++p) {
            T a[9], a1[9];
            AhStore<T>::load(cb + (size_t)(p * 2) * 9 * Vp, (int)Vp, s, a);
            AhStore<T>::load(cb + (size_t)(p * 2 + 1) * 9 * Vp, (int)Vp, s, a1);
#pragma unroll
            for (int k = 0; k < 9; ++k) a[k] += a1[k];
            if (traceless) {
                const T tr = (a[0] + a[1] + a[2]) * (T(1) / T(3));
                a[0] -= tr; a[1] -= tr; a[2] -= tr;
            }
            te += a[0] * a[0] + a[1] * a[1] + a[2] * a[2] +
                  T(2) * (a[3] * a[3] + a[4] * a[4] + a[5] * a[5] + a[6] * a[6] + a[7] * a[7] + a[8] * a[8]);
            if (p & 1) {
                const T d = a0[0] * a[0] + a0[1] * a[1] + a0[2] * a[2] +
                            T(2) * (a0[3] * a[3] + a0[4] * a[4] + a0[5] * a[5] + a0[6] * a[6] + a0[7] * a[7] + a0[8] * a[8]);
                tq += (p == 3) ? -d : d;
            } else {
#pragma unroll
                for (int k = 0; k < 9; ++k) a0[k] = a[k];
            }
            tp += __ldg(cb + (size_t)(108 + p) * Vp + s);
        }
        e = (double)te;
        q = (double)tq;
        pl = (double)tp;
    }
    e = warp_sum(e);
    q = warp_sum(q);
    pl = warp_sum(pl);
    if (lane == 0) {
        red[warp][0] = e;
        red[warp][1] = q;
        red[warp][2] = pl;
    }
    __syncthreads();
    const int nb = (c.V + kMeasureSites - 1) / kMeasureSites;
    if (threadIdx.x == 0) {
        double v[3] = {0, 0, 0};
#pragma unroll
        for (int i = 0; i < kMeasureSites / 32; ++i)
#pragma unroll
            for (int k = 0; k < 3; ++k) v[k] += red[i][k];
        double* o = partial + (size_t)blockIdx.x * kPartials;
        o[0] = v[0];
        o[1] = v[1];
        o[2] = v[2];
        if (LAST) {
            __threadfence();
            last = atomicAdd(reinterpret_cast<unsigned*>(c.x_off), 1u) == (unsigned)(nb - 1);
        }
    }
    if (!LAST) return;
    __syncthreads();
    if (!last) return;
    const int lo = nb * warp / 4, hi = nb * (warp + 1) / 4;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double v = sum_partials(partial + (size_t)(c.blk0 + lo) * kPartials, hi - lo, k, lane);
        if (lane == 0) red[warp][k] = v;
    }
    __syncthreads();
    if (threadIdx.x == 0)
        write_record(c, (red[0][0] + red[1][0]) + (red[2][0] + red[3][0]), (red[0][1] + red[1][1]) + (red[2][1] + red[3][1]),
                     (red[0][2] + red[1][2]) + (red[2][2] + red[3][2]), obs);
}

// One block per configuration of the launch: the sums over its partials, by four warps each.
template <int CAP>
__global__ void __launch_bounds__(384)
k_reduce(const __grid_constant__ BatchT<CAP> B, const double* __restrict__ partial, double* __restrict__ obs) {
    __shared__ double red[12];
    const CfgDesc& c = B.c[blockIdx.x];
    const int nb = (c.V + kMeasureSites - 1) / kMeasureSites, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int lo = nb * (warp & 3) / 4, hi = nb * ((warp & 3) + 1) / 4;
    const double v = sum_partials(partial + (size_t)(c.blk0 + lo) * kPartials, hi - lo, warp >> 2, lane);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (threadIdx.x == 0)
        write_record(c, (red[0] + red[1]) + (red[2] + red[3]), (red[4] + red[5]) + (red[6] + red[7]),
                     (red[8] + red[9]) + (red[10] + red[11]), obs);
}

// q(x0, t) (Sec. 4): the charge density summed over the slab x_dir = x of each configuration, FP64 sums in a
// fixed order.  A slab is cut into chunks of kSliceSites sites, one block and one site per thread each
// (the launch descriptor has L[dir] slice_chunks(n_slab) blocks per configuration), so that a few long slabs still
// fill the chip: with one block per slab, 72 slabs of 5184 sites left half the SMs idle and took 75 us, now 29 and 4
// for the sums (the halves' 161 MB at 6.7 TB/s take 24); tgf_measure_slices of 2 x 12x12x36x36 in FP32 183 -> 139 us
// (127 with the halves of planes.cuh).
// A slab of one chunk is finished here; the
// others leave a partial sum per block (x_off: the configuration's first one) for k_slice_reduce.
// q_out[cfg_index * q_stride + x] with cfg_index = c.o_off.
template <class T, int CAP>
__global__ void __launch_bounds__(kSliceSites)
k_slice_charge(const __grid_constant__ BatchT<CAP> B, const T* __restrict__ clov, int dir, double* __restrict__ q_out,
               int q_stride, double* __restrict__ partial, int traceless) {
    __shared__ double red[kSliceSites / 32];
    const int ci = find_cfg(B, blockIdx.x);
    const CfgDesc& c = B.c[ci];
    const int n_slab = c.V / c.L[dir], nch = slice_chunks(n_slab);
    const int b = blockIdx.x - c.blk0, x = b / nch, j = (b - x * nch) * kSliceSites + threadIdx.x;
    double q = 0.0;
    if (j < n_slab) {
        // the slab's sites: high st[dir+1] + x st[dir] + low with j = high st[dir] + low
        const int st = c.st[dir], high = j / st;
        const int s = high * c.st[dir + 1] + x * st + (j - high * st);
        const T* cb = clov + c.m_off;
        const size_t Vp = (size_t)c.Vp;
        T a0[9], tq = T(0);
#pragma unroll
        for (int p = 0; p < 6; ++p) {
            T a[9], a1[9];
            AhStore<T>::load(cb + (size_t)(p * 2) * 9 * Vp, (int)Vp, s, a);
            AhStore<T>::load(cb + (size_t)(p * 2 + 1) * 9 * Vp, (int)Vp, s, a1);
#pragma unroll
            for (int k = 0; k < 9; ++k) a[k] += a1[k];
            if (traceless) {
                const T tr = (a[0] + a[1] + a[2]) * (T(1) / T(3));
                a[0] -= tr; a[1] -= tr; a[2] -= tr;
            }
            if (p & 1) {
                const T d = a0[0] * a[0] + a0[1] * a[1] + a0[2] * a[2] +
                            T(2) * (a0[3] * a[3] + a0[4] * a[4] + a0[5] * a[5] + a0[6] * a[6] + a0[7] * a[7] + a0[8] * a[8]);
                tq += (p == 3) ? -d : d;
            } else {
#pragma unroll
                for (int k = 0; k < 9; ++k) a0[k] = a[k];
            }
        }
        q = (double)tq;
    }
    q = warp_sum(q);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = q;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
#pragma unroll
        for (int i = 0; i < kSliceSites / 32; ++i) v += red[i];
        if (nch == 1) q_out[(size_t)c.o_off * q_stride + x] = v * kSliceUnit;
        else partial[c.x_off + b] = v;
    }
}

// One warp per slab of more than one chunk: its partial sums in a fixed order (blocks: L[dir] per configuration).
template <int CAP>
__global__ void __launch_bounds__(32)
k_slice_reduce(const __grid_constant__ BatchT<CAP> B, int dir, double* __restrict__ q_out, int q_stride,
               const double* __restrict__ partial) {
    const int ci = find_cfg(B, blockIdx.x);
    const CfgDesc& c = B.c[ci];
    const int nch = slice_chunks(c.V / c.L[dir]);
    if (nch == 1) return;
    const int x = blockIdx.x - c.blk0;
    double v = 0.0;
    for (int i = threadIdx.x; i < nch; i += 32) v += partial[c.x_off + (int64_t)x * nch + i];
    v = warp_sum(v);
    if (threadIdx.x == 0) q_out[(size_t)c.o_off * q_stride + x] = v * kSliceUnit;
}

template <class T, int CAP>
static void slices_cap(const Batch& B, const Batch& R, const void* clov, int dir, double* q, int q_stride, double* partial,
                       unsigned flags, cudaStream_t st) {
    BatchT<CAP> b, r;
    b.ncfg = r.ncfg = B.ncfg;
    b.nblk = B.nblk;
    r.nblk = R.nblk;
    for (int i = 0; i < B.ncfg; ++i) {
        b.c[i] = B.c[i];
        r.c[i] = R.c[i];
    }
    k_slice_charge<T, CAP><<<b.nblk, kSliceSites, 0, st>>>(b, (const T*)clov, dir, q, q_stride, partial, (int)(flags & 1u));
    if (b.nblk > r.nblk) k_slice_reduce<CAP><<<r.nblk, 32, 0, st>>>(r, dir, q, q_stride, partial);
}

void launch_slice_charge(int prec, unsigned flags, const Batch& B, const Batch& R, const void* clov, int dir, double* q,
                         int q_stride, double* partial, cudaStream_t st) {
    const bool small = B.ncfg <= kSmallCap;
    if (prec == P64) small ? slices_cap<double, kSmallCap>(B, R, clov, dir, q, q_stride, partial, flags, st)
                           : slices_cap<double, kMaxCfg>(B, R, clov, dir, q, q_stride, partial, flags, st);
    else small ? slices_cap<float, kSmallCap>(B, R, clov, dir, q, q_stride, partial, flags, st)
               : slices_cap<float, kMaxCfg>(B, R, clov, dir, q, q_stride, partial, flags, st);
}

constexpr int kLastBlocks = 608;  // up to this many blocks (4 per SM) the last one reduces

template <class T, int CAP>
static void sum_cap(unsigned flags, const Batch& B, const void* clov, double* partial, double* obs, cudaStream_t st) {
    BatchT<CAP> b;
    b.ncfg = B.ncfg;
    b.nblk = B.nblk;
    for (int i = 0; i < B.ncfg; ++i) b.c[i] = B.c[i];
    if (B.nblk <= kLastBlocks) {
        k_clover_sum<T, CAP, true><<<B.nblk, kMeasureSites, 0, st>>>(b, (const T*)clov, partial, obs, (int)(flags & 1u));
    } else {
        k_clover_sum<T, CAP, false><<<B.nblk, kMeasureSites, 0, st>>>(b, (const T*)clov, partial, obs, (int)(flags & 1u));
        k_reduce<CAP><<<B.ncfg, 384, 0, st>>>(b, partial, obs);
    }
}

void launch_clover_sum(int prec, unsigned flags, const Batch& B, const void* clov, double* partial, double* obs,
                       cudaStream_t st) {
    if (B.ncfg <= kSmallCap) {
        if (prec == P64) sum_cap<double, kSmallCap>(flags, B, clov, partial, obs, st);
        else sum_cap<float, kSmallCap>(flags, B, clov, partial, obs, st);
    } else {
        if (prec == P64) sum_cap<double, kMaxCfg>(flags, B, clov, partial, obs, st);
        else sum_cap<float, kMaxCfg>(flags, B, clov, partial, obs, st);
    }
}

TGF_CHECK_WORD(measure)

}  // namespace tgf
