// stage64.cu -- the RK3 stage kernels in double precision (stage64.cuh).
#include "stage64.cuh"

namespace tgf {

namespace {

// Up to this many blocks a launch takes three threads per link (WIDE): one block of 384 threads per SM.  Measured on
// 3-step flows of n x 4x4x12x12 (72 n blocks), 128 and 384 threads: n = 1 379 and 329 us, n = 2 393 and 360 us,
// n = 3 488 and 585 us.
constexpr int kWideBlocks64 = 152;

template <int STAGE, int MODE, int CAP, bool WIDE>
void launch_cap(const Batch& B, const double* w_in, double* w_out, double* acc, double* clov, cudaStream_t st, int grid) {
    const int g = (grid > 0 && grid < B.nblk) ? grid : B.nblk;
    if constexpr (CAP == kMaxCfg) {
        k_stage64<STAGE, MODE, kMaxCfg, WIDE><<<g, stage64_threads(MODE, WIDE), 0, st>>>(B, w_in, w_out, acc, clov);
    } else {
        BatchT<CAP> b;
        b.ncfg = B.ncfg;
        b.nblk = B.nblk;
        for (int i = 0; i < B.ncfg; ++i) b.c[i] = B.c[i];
        k_stage64<STAGE, MODE, CAP, WIDE><<<g, stage64_threads(MODE, WIDE), 0, st>>>(b, w_in, w_out, acc, clov);
    }
}

template <int STAGE, int MODE>
void launch_m(const Batch& B, const double* w_in, double* w_out, double* acc, double* clov, cudaStream_t st, int grid) {
    if (B.nblk <= kWideBlocks64) {
        if (B.ncfg <= kSmallCap) launch_cap<STAGE, MODE, kSmallCap, true>(B, w_in, w_out, acc, clov, st, grid);
        else launch_cap<STAGE, MODE, kMaxCfg, true>(B, w_in, w_out, acc, clov, st, grid);
    } else {
        if (B.ncfg <= kSmallCap) launch_cap<STAGE, MODE, kSmallCap, false>(B, w_in, w_out, acc, clov, st, grid);
        else launch_cap<STAGE, MODE, kMaxCfg, false>(B, w_in, w_out, acc, clov, st, grid);
    }
}

}  // namespace

void launch_stage64(int stage, int mode, const Batch& B, const double* w_in, double* w_out, double* acc, double* clov,
                    cudaStream_t st, int grid) {
    if (mode == 2) launch_m<1, 2>(B, w_in, w_out, acc, clov, st, grid);
    else if (stage == 1 && mode == 1) launch_m<1, 1>(B, w_in, w_out, acc, clov, st, grid);
    else if (stage == 1) launch_m<1, 0>(B, w_in, w_out, acc, clov, st, grid);
    else if (stage == 2) launch_m<2, 0>(B, w_in, w_out, acc, clov, st, grid);
    else launch_m<3, 0>(B, w_in, w_out, acc, clov, st, grid);
}

TGF_CHECK_WORD(stage64)

}  // namespace tgf
