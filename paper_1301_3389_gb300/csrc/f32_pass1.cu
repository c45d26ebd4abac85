// Launchers of pass 1 in float32 (f32_pass.cuh), one instantiation per multiple of 16 of
// the rank.
#include "f32_pass.cuh"

namespace dna {
namespace f2 {

template <int RPT, bool WITH_B, int SG>
__global__ void __launch_bounds__(NT, 2)
    k_pass1_f2(View v, float* __restrict__ Apart, float* __restrict__ Bpart, int64_t s_per,
               int* __restrict__ status) {
    pdl_wait();
    extern __shared__ __align__(16) float smem_f2[];
    pass1_tile<RPT, WITH_B, SG>(v, Apart, Bpart, s_per, status, blockIdx.x, blockIdx.y, smem_f2);
}

template <int RPT, bool WITH_B, int SG>
static int launch(const View& v, float* A, float* B, int splits, int64_t s_per, int* status,
                  cudaStream_t st) {
    auto k = k_pass1_f2<RPT, WITH_B, SG>;
    const size_t smem = Pass1<RPT, WITH_B, SG>::smem;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
        cudaSuccess)
        return DNA_ERR_CUDA;
    const dim3 grid((unsigned)((v.O + OB - 1) / OB), (unsigned)splits);
    dna::launch_pdl(k, grid, dim3(NT), smem, st, v, A, B, s_per, status);
    return after_launch();
}

template <int RPT>
static int pick(const View& v, float* A, float* B, int splits, int64_t s_per, bool with_b,
                bool ascending, int* status, cudaStream_t st) {
    constexpr int SG = s_groups(RPT);
    if (ascending && SG > 1)
        return with_b ? launch<RPT, true, 1>(v, A, B, splits, s_per, status, st)
                      : launch<RPT, false, 1>(v, A, B, splits, s_per, status, st);
    return with_b ? launch<RPT, true, SG>(v, A, B, splits, s_per, status, st)
                  : launch<RPT, false, SG>(v, A, B, splits, s_per, status, st);
}

int pass1(const View& v, float* A, float* B, int splits, int64_t s_per, bool with_b,
          bool ascending, int* status, cudaStream_t st) {
    switch ((v.R + 15) / 16) {
        case 1: return pick<1>(v, A, B, splits, s_per, with_b, ascending, status, st);
        case 2: return pick<2>(v, A, B, splits, s_per, with_b, ascending, status, st);
        case 3: return pick<3>(v, A, B, splits, s_per, with_b, ascending, status, st);
        case 4: return pick<4>(v, A, B, splits, s_per, with_b, ascending, status, st);
        case 5: return pick<5>(v, A, B, splits, s_per, with_b, ascending, status, st);
        case 6: return pick<6>(v, A, B, splits, s_per, with_b, ascending, status, st);
        case 7: return pick<7>(v, A, B, splits, s_per, with_b, ascending, status, st);
        case 8: return pick<8>(v, A, B, splits, s_per, with_b, ascending, status, st);
        default: return DNA_ERR_UNSUPPORTED;
    }
}

}  // namespace f2
}  // namespace dna
