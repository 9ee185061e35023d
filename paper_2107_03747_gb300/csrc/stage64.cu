// stage64.cu -- the RK3 stage kernels in double precision (stage64.cuh).
#include "stage64.cuh"

namespace tgf {

namespace {

template <int STAGE, int MODE, int CAP>
void launch_cap(const Batch& B, const double* w_in, double* w_out, double* acc, double* clov, cudaStream_t st, int grid) {
    const int g = (grid > 0 && grid < B.nblk) ? grid : B.nblk;
    if constexpr (CAP == kMaxCfg) {
        k_stage64<STAGE, MODE, kMaxCfg><<<g, 128, 0, st>>>(B, w_in, w_out, acc, clov);
    } else {
        BatchT<CAP> b;
        b.ncfg = B.ncfg;
        b.nblk = B.nblk;
        for (int i = 0; i < B.ncfg; ++i) b.c[i] = B.c[i];
        k_stage64<STAGE, MODE, CAP><<<g, 128, 0, st>>>(b, w_in, w_out, acc, clov);
    }
}

template <int STAGE, int MODE>
void launch_m(const Batch& B, const double* w_in, double* w_out, double* acc, double* clov, cudaStream_t st, int grid) {
    if (B.ncfg <= kSmallCap) launch_cap<STAGE, MODE, kSmallCap>(B, w_in, w_out, acc, clov, st, grid);
    else launch_cap<STAGE, MODE, kMaxCfg>(B, w_in, w_out, acc, clov, st, grid);
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
