// Launchers of pass 2 and d_KL's column sums in float32 (f32_pass.cuh).
#include "f32_pass.cuh"

namespace dna {
namespace f2 {

template <int RPT, int NC, bool FULL>
__global__ void __launch_bounds__(NT, 2)
    k_pass2_f2(View v, const float* __restrict__ X0, const float* __restrict__ X1, int64_t xr,
               int64_t xo, double* __restrict__ dpart, int64_t s_per, int* __restrict__ status) {
    extern __shared__ __align__(16) float smem_f2[];
    pass2_tile<RPT, NC, FULL>(v, X0, X1, xr, xo, dpart, s_per, status, blockIdx.x, blockIdx.y,
                              smem_f2);
}

template <int RPT, int NC, bool FULL>
static int launch(const View& v, const float* X0, const float* X1, int64_t xr, int64_t xo,
                  double* dpart, int splits, int64_t s_per, int* status, cudaStream_t st) {
    auto k = k_pass2_f2<RPT, NC, FULL>;
    const size_t smem = Pass2<RPT, NC>::smem;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
        cudaSuccess)
        return DNA_ERR_CUDA;
    const dim3 grid((unsigned)((v.O + OB - 1) / OB), (unsigned)splits);
    k<<<grid, NT, smem, st>>>(v, X0, X1, xr, xo, dpart, s_per, status);
    return after_launch();
}

template <int NC, bool FULL>
static int any_rank(const View& v, const float* X0, const float* X1, int64_t xr, int64_t xo,
                    double* dpart, int splits, int64_t s_per, int* status, cudaStream_t st) {
    switch ((v.R + 15) / 16) {
        case 1: return launch<1, NC, FULL>(v, X0, X1, xr, xo, dpart, splits, s_per, status, st);
        case 2: return launch<2, NC, FULL>(v, X0, X1, xr, xo, dpart, splits, s_per, status, st);
        case 3: return launch<3, NC, FULL>(v, X0, X1, xr, xo, dpart, splits, s_per, status, st);
        case 4: return launch<4, NC, FULL>(v, X0, X1, xr, xo, dpart, splits, s_per, status, st);
        case 5: return launch<5, NC, FULL>(v, X0, X1, xr, xo, dpart, splits, s_per, status, st);
        case 6: return launch<6, NC, FULL>(v, X0, X1, xr, xo, dpart, splits, s_per, status, st);
        case 7: return launch<7, NC, FULL>(v, X0, X1, xr, xo, dpart, splits, s_per, status, st);
        case 8: return launch<8, NC, FULL>(v, X0, X1, xr, xo, dpart, splits, s_per, status, st);
        default: return DNA_ERR_UNSUPPORTED;
    }
}

int pass2(const View& v, const float* Xmu, const float* Xdna, double* dpart, int splits,
          int64_t s_per, int* status, cudaStream_t st) {
    return any_rank<2, false>(v, Xmu, Xdna, v.O, 1, dpart, splits, s_per, status, st);
}

int pass2_one(const View& v, const float* X, double* dpart, int splits, int64_t s_per,
              int* status, cudaStream_t st) {
    return any_rank<1, false>(v, X, X, v.O, 1, dpart, splits, s_per, status, st);
}

int kl_columns(const View& v, double* dpart, int splits, int64_t s_per, int* status,
               cudaStream_t st) {
    const float* X = static_cast<const float*>(v.X);
    return any_rank<1, true>(v, X, X, v.xr, v.xo, dpart, splits, s_per, status, st);
}

}  // namespace f2
}  // namespace dna
