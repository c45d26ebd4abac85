// Launchers of pass 2 and d_KL's column sums in float32 (f32_pass.cuh).
#include "f32_pass.cuh"

namespace dna {
namespace f2 {

template <int RPT, int NC, bool FULL>
__global__ void __launch_bounds__(NT, 2)
    k_pass2_f2(View v, const float* __restrict__ X0, const float* __restrict__ X1, int64_t xr,
               int64_t xo, double* __restrict__ dpart, int64_t s_per, int* __restrict__ status) {
    pdl_wait();
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
    dna::launch_pdl(k, grid, dim3(NT), smem, st, v, X0, X1, xr, xo, dpart, s_per, status);
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

// Gradient of eq. 1 with respect to V: dV(s, o) = scale log(v / z) where v > 0, else 0.  A
// CTA owns a 64 x 64 tile (one load of x and y each): bound by the tile's operand loads and
// by V in and dV out (N=1024 T=4096 R=64: 34 us with 4 x 4 scalar tiles, 26 now).
template <int RPT>
__global__ void __launch_bounds__(NT, 2)
    k_grad_v_f2(View v, float scale, float* __restrict__ dV, int64_t ldd,
                int* __restrict__ status) {
    pdl_wait();
    using H = Tiles<RPT>;
    extern __shared__ __align__(16) float smem_f2[];
    float* Xs = smem_f2;
    float* Ys = Xs + H::X;
    const float* __restrict__ V = static_cast<const float*>(v.V);
    const int64_t o0 = (int64_t)blockIdx.x * OB, s0 = (int64_t)blockIdx.y * SB;
    const ZPos zp = z_pos();
    load_x<H::RB>(Xs, static_cast<const float*>(v.X), v.xr, v.xo, o0, v.O, v.R);
    load_y<H::RB>(Ys, static_cast<const float*>(v.Y), v.ys, v.yr, s0, v.S, v.R);
    cp_commit();
    const bool wide = v_wide(v), wide_d = ((ldd | v.O) & 3) == 0 &&
                                          (reinterpret_cast<uintptr_t>(dV) & 15) == 0;
    const int64_t o = o0 + 4 * zp.ol;
    float vv[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) load_v(v, V, wide, s0 + zp.sl + 16 * i, v.S, o, vv[i]);
    cp_wait<0>();
    __syncthreads();
    u64 z[1][4][2];
    z_tile<H::RB, 1>(Ys, Xs, zp, (int)((v.R + 3) / 4), z);
    int bad = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int64_t s = s0 + zp.sl + 16 * i;
        if (s >= v.S) continue;
        const float2 z0 = unpack2(z[0][i][0]), z1 = unpack2(z[0][i][1]);
        const float zz[4] = {z0.x, z0.y, z1.x, z1.y};
        float g[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const bool pos = vv[i][j] > 0.f;
            bad |= pos && !(zz[j] > 0.f) ? 1 : 0;
            g[j] = pos && zz[j] > 0.f ? scale * logf(vv[i][j] / zz[j]) : 0.f;
        }
        float* p = dV + s * ldd + o;
        if (wide_d) {
            if (o < v.O) *reinterpret_cast<float4*>(p) = make_float4(g[0], g[1], g[2], g[3]);
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (o + j < v.O) p[j] = g[j];
        }
    }
    if (bad) atomicOr(status, STATUS_NONFINITE);
}

template <int RPT>
static int launch_grad(const View& v, float scale, float* dV, int64_t ldd, int* status,
                       cudaStream_t st) {
    auto k = k_grad_v_f2<RPT>;
    const size_t smem = sizeof(float) * (Tiles<RPT>::X + Tiles<RPT>::Y);
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
        cudaSuccess)
        return DNA_ERR_CUDA;
    const dim3 grid((unsigned)((v.O + OB - 1) / OB), (unsigned)((v.S + SB - 1) / SB));
    dna::launch_pdl(k, grid, dim3(NT), smem, st, v, scale, dV, ldd, status);
    return after_launch();
}

int grad_v(const View& v, float scale, float* dV, int64_t ldd, int* status, cudaStream_t st) {
    switch ((v.R + 15) / 16) {
        case 1: return launch_grad<1>(v, scale, dV, ldd, status, st);
        case 2: return launch_grad<2>(v, scale, dV, ldd, status, st);
        case 3: return launch_grad<3>(v, scale, dV, ldd, status, st);
        case 4: return launch_grad<4>(v, scale, dV, ldd, status, st);
        case 5: return launch_grad<5>(v, scale, dV, ldd, status, st);
        case 6: return launch_grad<6>(v, scale, dV, ldd, status, st);
        case 7: return launch_grad<7>(v, scale, dV, ldd, status, st);
        case 8: return launch_grad<8>(v, scale, dV, ldd, status, st);
        default: return DNA_ERR_UNSUPPORTED;
    }
}

}  // namespace f2
}  // namespace dna
