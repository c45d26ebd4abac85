// Host launchers for the SIMT kernels (instantiated for float and double).
#pragma once

#include <algorithm>
#include <type_traits>

#include "glue_kernels.cuh"
#include "simt_kernels.cuh"
#include "sparse_kernels.cuh"

namespace dna {

namespace simt {

template <typename Tp> constexpr int rblock_for(int64_t R) {
    return sizeof(Tp) == 4 ? (R <= 32 ? 32 : (R <= 64 ? 64 : 128)) : (R <= 32 ? 32 : 64);
}

inline int launch_status() { return after_launch(); }

// Opts a kernel in to its dynamic shared memory.  The limit without opting in is 48 KB of
// static and dynamic memory together, and the kernels here have up to 12 KB of static arrays.
template <typename Kern>
inline int prep_smem(Kern k, size_t bytes) {
    static_assert(sizeof(Kern) > 0, "");
    if (bytes > 32 * 1024) {
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) !=
            cudaSuccess)
            return DNA_ERR_CUDA;
    }
    return DNA_OK;
}

template <typename Tp, int RB>
int pass1_rb(const View& v, Tp* A, Tp* B, int splits, int64_t s_per, bool with_b, int* status,
             cudaStream_t st, double* dcur) {
    const size_t smem = Pass1Cfg<Tp, RB>::smem;
    dim3 grid((unsigned)((v.O + OB - 1) / OB), (unsigned)((v.R + RB - 1) / RB), (unsigned)splits);
    auto launch = [&](auto k) {
        if (prep_smem(k, smem)) return DNA_ERR_CUDA;
        // float32 above rank 128: a plain launch.  Its plan fills the SMs in one wave of two CTAs
        // each, which took longer where programmatic serialisation let it start beside the
        // operand kernel: N=1000 T=1200, DNA iteration at R = 129 731 us without any, 782 with
        // it here, 706 as it is (with it in the other kernels); MU at R = 129 289, 340, 282;
        // DNA at R = 512 1602, 1559, 1566
        if (sizeof(Tp) == 4 && v.R > f2::MAX_R)
            k<<<grid, NT, smem, st>>>(v, A, B, s_per, status, dcur);
        else
            dna::launch_pdl(k, grid, dim3(NT), smem, st, v, A, B, s_per, status, dcur);
        return launch_status();
    };
    // float32 at ranks up to 128 comes here for descent selection only, which needs B
    if constexpr (sizeof(Tp) == 8 || RB == 128)
        if (!with_b) return launch(k_pass1<Tp, RB, false>);
    return with_b ? launch(k_pass1<Tp, RB, true>) : DNA_ERR_UNSUPPORTED;
}

template <typename Tp, int RB, int NC, bool FULL>
int pass2_rb(const View& v, const Tp* X0, const Tp* X1, int64_t xr, int64_t xo, double* dpart,
             int splits, int64_t s_per, int* status, cudaStream_t st) {
    const size_t smem = Pass2Cfg<Tp, RB, NC>::smem;
    auto k = k_pass2<Tp, RB, NC, FULL>;
    if (prep_smem(k, smem)) return DNA_ERR_CUDA;
    dim3 grid((unsigned)((v.O + OB - 1) / OB), (unsigned)splits);
    dna::launch_pdl(k, grid, dim3(NT), smem, st, v, X0, X1, xr, xo, dpart, s_per, status);
    return launch_status();
}

template <typename Tp, int NC, bool FULL>
int pass2_any(const View& v, const Tp* X0, const Tp* X1, int64_t xr, int64_t xo, double* dpart,
              int splits, int64_t s_per, int* status, cudaStream_t st) {
    // float32 at ranks up to f2::MAX_R runs in f32_pass.cuh
    if constexpr (sizeof(Tp) == 4)
        return pass2_rb<Tp, 128, NC, FULL>(v, X0, X1, xr, xo, dpart, splits, s_per, status, st);
    else if (rblock_for<Tp>(v.R) == 32)
        return pass2_rb<Tp, 32, NC, FULL>(v, X0, X1, xr, xo, dpart, splits, s_per, status, st);
    else
        return pass2_rb<Tp, 64, NC, FULL>(v, X0, X1, xr, xo, dpart, splits, s_per, status, st);
}

template <typename Tp, int RB>
int occupancy_pass1() {
    int nb = 0;
    auto k = k_pass1<Tp, RB, true>;
    if (prep_smem(k, Pass1Cfg<Tp, RB>::smem)) return 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, NT, Pass1Cfg<Tp, RB>::smem) !=
        cudaSuccess)
        return 1;
    return nb > 0 ? nb : 1;
}

template <typename Tp, int RB>
int occupancy_pass2() {
    int nb = 0;
    auto k = k_pass2<Tp, RB, 2, false>;
    if (prep_smem(k, Pass2Cfg<Tp, RB, 2>::smem)) return 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, NT, Pass2Cfg<Tp, RB, 2>::smem) !=
        cudaSuccess)
        return 1;
    return nb > 0 ? nb : 1;
}

}  // namespace simt

namespace simt {
// sum over i < n of M(i, r) + reg -> out[r], M(i, r) at M[i * si + r * sr]: one CTA per r
// when rows are contiguous, else a two-level column sum through `work`
// (at least FSUM_SPLITS * R float64).
template <typename Tp>
int factor_sums(const Tp* M, int64_t n, int64_t R, int64_t si, int64_t sr, double reg,
                double* out, double* work, cudaStream_t st) {
    if (sr != 1 && si == 1) {
        k_row_sums<Tp><<<(unsigned)R, 256, 0, st>>>(M, n, sr, reg, out, true);
        return launch_status();
    }
    const int64_t nsplit = std::max<int64_t>(1, std::min<int64_t>(FSUM_SPLITS, (n + 63) / 64));
    const int64_t rows_per = (n + nsplit - 1) / nsplit;
    dim3 blk(32, 8);
    dim3 grid((unsigned)((R + 31) / 32), (unsigned)nsplit);
    k_colsum_part<Tp><<<grid, blk, 0, st>>>(M, n, R, si, sr, rows_per, work);
    if (launch_status()) return DNA_ERR_CUDA;
    k_colsum_final<<<(unsigned)((R + 31) / 32), dim3(32, 32), 0, st>>>(work, (int)nsplit, R, reg, out,
                                                                      true);
    return launch_status();
}
}  // namespace simt

template <typename Tp>
int Simt<Tp>::factor_sums_y(const View& v, double reg, double* out, double* work,
                            cudaStream_t st) {
    return simt::factor_sums<Tp>(static_cast<const Tp*>(v.Y), v.S, v.R, v.ys, v.yr, reg, out,
                                 work, st);
}

template <typename Tp>
int Simt<Tp>::factor_sums_x(const View& v, double reg, double* out, double* work,
                            cudaStream_t st) {
    return simt::factor_sums<Tp>(static_cast<const Tp*>(v.X), v.O, v.R, v.xo, v.xr, reg, out,
                                 work, st);
}

template <typename Tp>
int Simt<Tp>::rescale(const View& v, const double* f, cudaStream_t st) {
    const int64_t rgroups = (v.R + 7) / 8;
    const int64_t longest = std::max(v.O, v.S);
    const int64_t bx = std::max<int64_t>(1, std::min<int64_t>(64, (longest + 511) / 512));
    dim3 grid((unsigned)bx, (unsigned)(2 * rgroups));
    simt::k_rescale<Tp><<<grid, dim3(32, 8), 0, st>>>(v, f, rgroups);
    return simt::launch_status();
}

template <typename Tp>
int Simt<Tp>::pass1(const View& v, Tp* A, Tp* B, int splits, int64_t s_per, bool with_b,
                    int* status, cudaStream_t st, double* dcur, bool ascending) {
    if constexpr (sizeof(Tp) == 4)
        if (v.R <= f2::MAX_R && !dcur)
            return f2::pass1(v, A, B, splits, s_per, with_b, ascending, status, st);
    switch (simt::rblock_for<Tp>(v.R)) {
        case 32: return simt::pass1_rb<Tp, 32>(v, A, B, splits, s_per, with_b, status, st, dcur);
        case 64: return simt::pass1_rb<Tp, 64>(v, A, B, splits, s_per, with_b, status, st, dcur);
        default:
            if constexpr (sizeof(Tp) == 4)
                return simt::pass1_rb<Tp, 128>(v, A, B, splits, s_per, with_b, status, st, dcur);
            return DNA_ERR_UNSUPPORTED;
    }
}

template <typename Tp>
int Simt<Tp>::candidates(const View& v, const double* c, const Tp* A, const Tp* B, int splits,
                         Tp* Xmu, Tp* Xdna, double eps, double alpha, cudaStream_t st) {
    simt::k_candidates<Tp><<<(unsigned)((v.O + 31) / 32), dim3(32, 8), 0, st>>>(
        v, c, A, B, splits, Xmu, Xdna, (Tp)eps, (Tp)alpha);
    return simt::launch_status();
}

template <typename Tp>
int Simt<Tp>::mu_apply(const View& v, const double* c, const Tp* A, int splits, cudaStream_t st) {
    simt::k_mu_apply<Tp><<<(unsigned)((v.O + 127) / 128), 128, 0, st>>>(v, c, A, splits);
    return simt::launch_status();
}

template <typename Tp>
int Simt<Tp>::pass2(const View& v, const Tp* Xmu, const Tp* Xdna, double* dpart, int splits,
                    int64_t s_per, int* status, cudaStream_t st) {
    if constexpr (sizeof(Tp) == 4)
        if (v.R <= f2::MAX_R) return f2::pass2(v, Xmu, Xdna, dpart, splits, s_per, status, st);
    return simt::pass2_any<Tp, 2, false>(v, Xmu, Xdna, v.O, 1, dpart, splits, s_per, status, st);
}

template <typename Tp>
int Simt<Tp>::pass2_one(const View& v, const Tp* X, double* dpart, int splits, int64_t s_per,
                        int* status, cudaStream_t st) {
    if constexpr (sizeof(Tp) == 4)
        if (v.R <= f2::MAX_R) return f2::pass2_one(v, X, dpart, splits, s_per, status, st);
    return simt::pass2_any<Tp, 1, false>(v, X, X, v.O, 1, dpart, splits, s_per, status, st);
}

template <typename Tp>
int Simt<Tp>::select(const View& v, const Tp* Xmu, const Tp* Xdna, const double* dpart,
                     int splits, uint8_t* choice, double* dfin, double reg, cudaStream_t st) {
    simt::k_select<Tp><<<(unsigned)((v.O + 31) / 32), dim3(32, 8), 0, st>>>(
        v, Xmu, Xdna, dpart, splits, choice, dfin, reg);
    return simt::launch_status();
}

template <typename Tp>
int Simt<Tp>::kl_columns(const View& v, double* dpart, int splits, int64_t s_per, int* status,
                         cudaStream_t st) {
    if constexpr (sizeof(Tp) == 4)
        if (v.R <= f2::MAX_R) return f2::kl_columns(v, dpart, splits, s_per, status, st);
    const Tp* X = static_cast<const Tp*>(v.X);
    return simt::pass2_any<Tp, 1, true>(v, X, X, v.xr, v.xo, dpart, splits, s_per, status, st);
}

template <typename Tp>
int Simt<Tp>::grad_x(const View& v, const double* c, const Tp* A, int splits, double scale,
                     Tp* G, int64_t gr, int64_t go, cudaStream_t st) {
    const dim3 grid((unsigned)((v.O + 31) / 32), (unsigned)((v.R + 63) / 64));
    simt::k_grad_x<Tp><<<grid, dim3(32, 8), 0, st>>>(v, c, A, splits, scale, G, gr, go);
    return simt::launch_status();
}

namespace simt {
template <typename Tp, int RB>
int grad_v_rb(const View& v, double scale, Tp* dV, int64_t ldd, int* status, cudaStream_t st) {
    const size_t smem = (size_t)(2 * RB * LD) * sizeof(Tp);
    auto k = k_grad_v<Tp, RB>;
    if (prep_smem(k, smem)) return DNA_ERR_CUDA;
    dim3 grid((unsigned)((v.O + OB - 1) / OB), (unsigned)((v.S + SB - 1) / SB));
    dna::launch_pdl(k, grid, dim3(NT), smem, st, v, scale, dV, ldd, status);
    return launch_status();
}
}  // namespace simt

template <typename Tp>
int Simt<Tp>::grad_v(const View& v, double scale, Tp* dV, int64_t ldd, int* status,
                     cudaStream_t st) {
    if constexpr (sizeof(Tp) == 4) {
        if (v.R <= f2::MAX_R) return f2::grad_v(v, (float)scale, dV, ldd, status, st);
        return simt::grad_v_rb<Tp, 128>(v, scale, dV, ldd, status, st);
    } else {
        return v.R <= 32 ? simt::grad_v_rb<Tp, 32>(v, scale, dV, ldd, status, st)
                         : simt::grad_v_rb<Tp, 64>(v, scale, dV, ldd, status, st);
    }
}

namespace simt {
template <typename Tp, int RB>
int adj_gemm_rb(const View& v, const Tp* Abar, const Tp* Bbar, const double* vs, Tp* Hpart,
                int splits, int64_t s_per, Tp* Vbar, int64_t ldvb, int* status, cudaStream_t st) {
    const size_t smem = AdjCfg<Tp, RB>::smem;
    auto k = k_adj_gemm<Tp, RB>;
    if (prep_smem(k, smem)) return DNA_ERR_CUDA;
    dim3 grid((unsigned)((v.O + OB - 1) / OB), (unsigned)splits);
    dna::launch_pdl(k, grid, dim3(NT), smem, st, v, Abar, Bbar, vs, Hpart, Vbar, ldvb, s_per,
                    status);
    return launch_status();
}
}  // namespace simt

template <typename Tp>
int Simt<Tp>::adjoint_elem(const View& v, const double* c, const Tp* A, const Tp* B,
                           const uint8_t* choice, const Tp* Hbar1, Tp* Hbar0, Tp* Abar, Tp* Bbar,
                           double* vs, double eps, double alpha, cudaStream_t st, double* cpart) {
    simt::k_adj_elem<Tp><<<(unsigned)((v.O + 31) / 32), dim3(32, 8), 0, st>>>(
        v, c, A, B, choice, Hbar1, Hbar0, Abar, Bbar, vs, (Tp)eps, (Tp)alpha, cpart);
    return simt::launch_status();
}

template <typename Tp>
int Simt<Tp>::adjoint_h(const View& v, const Tp* Abar, const Tp* Bbar, const double* vs,
                        Tp* Hpart, int splits, int64_t s_per, Tp* Vbar, int64_t ldvb, int* status,
                        cudaStream_t st) {
    if constexpr (sizeof(Tp) == 4)
        return DNA_ERR_UNSUPPORTED;   // f32_adjoint.cu
    else if (simt::rblock_for<Tp>(v.R) == 32)
        return simt::adj_gemm_rb<Tp, 32>(v, Abar, Bbar, vs, Hpart, splits, s_per, Vbar, ldvb,
                                         status, st);
    else if (v.R <= 64)
        return simt::adj_gemm_rb<Tp, 64>(v, Abar, Bbar, vs, Hpart, splits, s_per, Vbar, ldvb,
                                         status, st);
    return DNA_ERR_UNSUPPORTED;
}

template <typename Tp>
int Simt<Tp>::adjoint_add(const View& v, const Tp* Hpart, int splits, Tp* Hbar0,
                          cudaStream_t st) {
    simt::k_adj_combine<Tp><<<(unsigned)((v.O + 31) / 32), dim3(32, 8), 0, st>>>(v, Hpart, splits,
                                                                                 Hbar0);
    return simt::launch_status();
}

namespace simt {
template <typename Tp, int RB>
int adj_wgrad_rb(const View& v, const Tp* Abar, const Tp* Bbar, Tp* Wpart, int wsplits,
                 int64_t o_per, int* status, cudaStream_t st) {
    const size_t smem = WgradCfg<Tp, RB>::smem;
    auto k = k_adj_wgrad<Tp, RB>;
    if (prep_smem(k, smem)) return DNA_ERR_CUDA;
    dim3 grid((unsigned)((v.S + SB - 1) / SB), (unsigned)wsplits);
    dna::launch_pdl(k, grid, dim3(NT), smem, st, v, Abar, Bbar, Wpart, o_per, status);
    return launch_status();
}
}  // namespace simt

template <typename Tp>
int Simt<Tp>::adjoint_w(const View& v, const Tp* Abar, const Tp* Bbar, const double* cpart,
                        Tp* Wpart, int wsplits, int64_t o_per, Tp* Wbar, int* status,
                        cudaStream_t st) {
    if constexpr (sizeof(Tp) == 4) {
        return DNA_ERR_UNSUPPORTED;   // f32_adjoint.cu
    } else {
        if (v.R > 64 || o_per % simt::OB) return DNA_ERR_UNSUPPORTED;
        const int e = v.R <= 32 ? simt::adj_wgrad_rb<Tp, 32>(v, Abar, Bbar, Wpart, wsplits, o_per,
                                                             status, st)
                                : simt::adj_wgrad_rb<Tp, 64>(v, Abar, Bbar, Wpart, wsplits, o_per,
                                                             status, st);
        if (e) return e;
        simt::k_adj_wcombine<Tp><<<(unsigned)((v.S + 31) / 32), dim3(32, 8), 0, st>>>(
            v, Wpart, wsplits, cpart, (v.O + 31) / 32, Wbar);
        return simt::launch_status();
    }
}

template <typename Tp>
int64_t Simt<Tp>::glue_parts(int64_t n) { return (n + glue::TO - 1) / glue::TO; }

template <typename Tp>
int Simt<Tp>::cand_fused(const View& v, const double* c, const Tp* A, const Tp* B, int splits,
                         Tp* Xmu, Tp* Xdna, double eps, double alpha, void* Xmk, void* Xdk,
                         int64_t rp, int64_t O_pad, int64_t plane, cudaStream_t st) {
    const bool bf = Xmk != nullptr;
    if (bf && (sizeof(Tp) != 4 || !Xdk || rp < v.R || rp % 2 != 0 || O_pad < v.O))
        return DNA_ERR_ARG;
    const unsigned grid = (unsigned)((bf ? O_pad : v.O) + glue::TO - 1) / glue::TO;
    if (cand_in_registers(v.R) && (!bf || rp <= 16 * (v.R <= 128 ? 8 : 16))) {
        // candidates of a thread in registers, at most 16 groups of r
        const int rs = v.R <= 128 ? 8 : 16;
        const int64_t rows = std::max<int64_t>((v.R + rs - 1) / rs, bf ? (rp + rs - 1) / rs : 0);
        const dim3 blk(32, (unsigned)rows);
        if (bf && rp % 8 != 0) return DNA_ERR_ARG;
        if (bf) {
            if constexpr (sizeof(Tp) == 4) {
                auto* bm = static_cast<glue::bf16*>(Xmk);
                auto* bd = static_cast<glue::bf16*>(Xdk);
                if (rs == 8)
                    dna::launch_pdl(glue::k_cand_reg<Tp, true, 8>, grid, blk, 0, st, v, c, A, B,
                                    splits, Xmu, Xdna, (Tp)eps, (Tp)alpha, bm, bd, rp, plane);
                else
                    dna::launch_pdl(glue::k_cand_reg<Tp, true, 16>, grid, blk, 0, st, v, c, A, B,
                                    splits, Xmu, Xdna, (Tp)eps, (Tp)alpha, bm, bd, rp, plane);
            }
        } else if (rs == 8) {
            dna::launch_pdl(glue::k_cand_reg<Tp, false, 8>, grid, blk, 0, st, v, c, A, B, splits,
                            Xmu, Xdna, (Tp)eps, (Tp)alpha, nullptr, nullptr, 0, 0);
        } else {
            dna::launch_pdl(glue::k_cand_reg<Tp, false, 16>, grid, blk, 0, st, v, c, A, B, splits,
                            Xmu, Xdna, (Tp)eps, (Tp)alpha, nullptr, nullptr, 0, 0);
        }
        return simt::launch_status();
    }
    if constexpr (sizeof(Tp) == 4) {   // float32 above the registers' ranks: R <= 512
        const unsigned cols = (unsigned)(((bf ? O_pad : v.O) + glue::CW_COLS - 1) / glue::CW_COLS);
        const size_t smem = glue::cand_wide_smem(rp, bf, plane != 0);
        auto k = bf ? glue::k_cand_wide<true> : glue::k_cand_wide<false>;
        if (v.R > 512 || (bf && rp > 512) || simt::prep_smem(k, smem)) return DNA_ERR_CUDA;
        dna::launch_pdl(k, cols, dim3(512), smem, st, v, c, A, B, splits, Xmu, Xdna, (Tp)eps,
                        (Tp)alpha, static_cast<glue::bf16*>(Xmk), static_cast<glue::bf16*>(Xdk),
                        rp, plane);
    } else {
        const size_t smem = glue::cand_smem<Tp>(v.R);
        auto k = glue::k_cand_fused<Tp>;
        if (simt::prep_smem(k, smem)) return DNA_ERR_CUDA;
        dna::launch_pdl(k, grid, dim3(32, glue::TY), smem, st, v, c, A, B, splits, Xmu, Xdna,
                        (Tp)eps, (Tp)alpha);
    }
    return simt::launch_status();
}

template <typename Tp>
bool Simt<Tp>::cand_in_registers(int64_t R) { return R <= (sizeof(Tp) == 8 ? 128 : 256); }

template <typename Tp>
int Simt<Tp>::split_sum(Tp* A, Tp* B, int64_t R, int64_t O, int splits, cudaStream_t st,
                        bool ascending) {
    if (splits <= 1) return DNA_OK;
    const int64_t n = R * O;
    const int vec = sizeof(Tp) == 4 && n % 4 == 0 ? 4 : 1;
    const int64_t work = n / vec;
    const unsigned ab = B ? 2 : 1;
    // above four splits the loads of one thread would be rounds of dependent latency
    if (splits > 4 && !ascending) {
        const dim3 grid((unsigned)((work + 31) / 32), ab);
        if constexpr (sizeof(Tp) == 4)
            if (vec == 4) {
                dna::launch_pdl(glue::k_split_sum_par<Tp, 4>, grid, dim3(32, 8), 0, st, A, B, n,
                                splits);
                return simt::launch_status();
            }
        dna::launch_pdl(glue::k_split_sum_par<Tp, 1>, grid, dim3(32, 8), 0, st, A, B, n, splits);
        return simt::launch_status();
    }
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((work + 255) / 256, 152 * 8));
    const dim3 grid((unsigned)blocks, ab);
    if constexpr (sizeof(Tp) == 4)
        if (vec == 4) {
            dna::launch_pdl(glue::k_split_sum<Tp, 4>, grid, dim3(256), 0, st, A, B, n, splits);
            return simt::launch_status();
        }
    dna::launch_pdl(glue::k_split_sum<Tp, 1>, grid, dim3(256), 0, st, A, B, n, splits);
    return simt::launch_status();
}

template <typename Tp>
int Simt<Tp>::select_fused(const View& v, const Tp* Xmu, const Tp* Xdna, const double* dpart,
                           int splits, uint8_t* choice, double* dfin, double* fpart,
                           double reg, cudaStream_t st, const double* dcur, int cur_splits) {
    const size_t smem = glue::select_smem<Tp>(v.R);
    auto k = glue::k_select_fused<Tp>;
    if (simt::prep_smem(k, smem)) return DNA_ERR_CUDA;
    dna::launch_pdl(k, dim3((unsigned)glue_parts(v.O)), dim3(32, 8), smem, st, v, Xmu, Xdna,
                    dpart, splits, choice, dfin, fpart, reg, dcur, cur_splits);
    return simt::launch_status();
}

template <typename Tp>
int Simt<Tp>::mu_fused(const View& v, const double* c, const Tp* A, int splits, double* fpart,
                       cudaStream_t st) {
    const size_t smem = glue::select_smem<Tp>(v.R);
    auto k = glue::k_mu_fused<Tp>;
    if (simt::prep_smem(k, smem)) return DNA_ERR_CUDA;
    dna::launch_pdl(k, dim3((unsigned)glue_parts(v.O)), dim3(32, 8), smem, st, v, c, A, splits,
                    fpart);
    return simt::launch_status();
}

template <typename Tp>
int Simt<Tp>::part_sums(const double* part, int64_t nparts, int64_t R, double reg, double* out,
                        cudaStream_t st, double* next) {
    if (R <= 1024)   // a CTA per r: latency of one load round and a tree, not of nparts / 32
        dna::launch_pdl(simt::k_colsum_small<0>, dim3((unsigned)R), dim3(256), 0, st, part,
                        (int)nparts, R, reg, out, true, next);
    else
        simt::k_colsum_final<<<(unsigned)((R + 31) / 32), dim3(32, 32), 0, st>>>(
            part, (int)nparts, R, reg, out, true, next);
    return simt::launch_status();
}

template <typename Tp>
int Simt<Tp>::scale_ops(const View& t, const double* f, bool xmul, void* Xk, void* Yk, void* Ytk,
                        void* Y2tk, int64_t rp, int64_t O_pad, int64_t S_pad, int64_t plane,
                        double* cpart, cudaStream_t st) {
    const bool bf = Xk != nullptr;
    if (bf && (sizeof(Tp) != 4 || !Yk || !Ytk || rp < t.R || O_pad < t.O || S_pad < t.S))
        return DNA_ERR_ARG;
    glue::OpsArgs a{};
    a.X = t.X; a.xr = t.xr; a.xo = t.xo; a.O = t.O;
    a.Y = const_cast<void*>(t.Y); a.ys = t.ys; a.yr = t.yr; a.S = t.S;
    a.R = t.R; a.f = f; a.xmul = xmul;
    a.Xk = static_cast<glue::bf16*>(Xk); a.Yk = static_cast<glue::bf16*>(Yk);
    a.Ytk = static_cast<glue::bf16*>(Ytk); a.Y2tk = static_cast<glue::bf16*>(Y2tk);
    a.rp = rp; a.O_pad = O_pad; a.S_pad = S_pad; a.plane = bf ? plane : 0; a.cpart = cpart;
    const int64_t rcov = bf ? rp : t.R, ocov = bf ? O_pad : t.O, scov = bf ? S_pad : t.S;
    const int rt = rcov <= 32 ? 32 : rcov <= 64 ? 64 : 128;   // values of r per tile
    a.tiles_r = (rcov + rt - 1) / rt;
    // without scaling and operands the X tiles have nothing to do
    a.xtiles_o = (f || bf) ? glue_parts(ocov) : 0;
    a.xtiles = a.xtiles_o * a.tiles_r;
    const int64_t ytiles = (f || bf || cpart) ? glue_parts(scov) * a.tiles_r : 0;
    const int64_t blocks = a.xtiles + ytiles;
    if (blocks == 0) return DNA_OK;
    if (rt == 32)
        dna::launch_pdl(glue::k_scale_ops<Tp, 32>, dim3((unsigned)blocks), dim3(32, 8), 0, st, a);
    else if (rt == 64)
        dna::launch_pdl(glue::k_scale_ops<Tp, 64>, dim3((unsigned)blocks), dim3(32, 8), 0, st, a);
    else
        dna::launch_pdl(glue::k_scale_ops<Tp, 128>, dim3((unsigned)blocks), dim3(32, 8), 0, st, a);
    return simt::launch_status();
}

template <typename Tp>
int Simt<Tp>::prepare_v(const Tp* V, int64_t N, int64_t T, int64_t ldv, Tp* Vt, int64_t ldvt,
                        double* colsum, double* rowsum, cudaStream_t st, double* part, Tp* Vc) {
    dim3 blk(32, 8);
    dim3 grid((unsigned)((T + 31) / 32), (unsigned)((N + 31) / 32));
    if (Vc && !part) return DNA_ERR_ARG;
    if (part) {   // one pass over V: transpose and per-tile sums, then the float64 totals
        double* colpart = part;                                // [ceil(N / 32)][T]
        double* rowpart = part + (size_t)((N + 31) / 32) * T;  // [ceil(T / 32)][N]
        simt::k_transpose_sums<Tp><<<grid, blk, 0, st>>>(V, N, T, ldv, Vt, ldvt, colpart, rowpart,
                                                         Vc);
        if (simt::launch_status()) return DNA_ERR_CUDA;
        simt::k_colsum_final<<<(unsigned)((T + 31) / 32), dim3(32, 32), 0, st>>>(
            colpart, (int)((N + 31) / 32), T, 0.0, colsum, false);
        if (simt::launch_status()) return DNA_ERR_CUDA;
        simt::k_colsum_final<<<(unsigned)((N + 31) / 32), dim3(32, 32), 0, st>>>(
            rowpart, (int)((T + 31) / 32), N, 0.0, rowsum, false);
        return simt::launch_status();
    }
    simt::k_transpose<Tp><<<grid, blk, 0, st>>>(V, N, T, ldv, Vt, ldvt);
    if (simt::launch_status()) return DNA_ERR_CUDA;
    // column sums of V: sum over n of V[n][t]  (coalesced across t)
    simt::k_factor_sums<Tp><<<(unsigned)((T + 31) / 32), blk, 0, st>>>(V, N, T, ldv, 1, 0.0, colsum,
                                                                             false);
    if (simt::launch_status()) return DNA_ERR_CUDA;
    // row sums of V: rows are contiguous
    simt::k_row_sums<Tp><<<(unsigned)N, 256, 0, st>>>(V, T, ldv, 0.0, rowsum, false);
    return simt::launch_status();
}

template <typename Tp>
int Simt<Tp>::pass1_blocks_per_sm(int64_t R) {
    switch (simt::rblock_for<Tp>(R)) {
        case 32: return simt::occupancy_pass1<Tp, 32>();
        case 64: return simt::occupancy_pass1<Tp, 64>();
        default:
            if constexpr (sizeof(Tp) == 4) return simt::occupancy_pass1<Tp, 128>();
            return 1;
    }
}

template <typename Tp>
int Simt<Tp>::pass2_blocks_per_sm(int64_t R) {
    if constexpr (sizeof(Tp) == 4)
        return simt::occupancy_pass2<Tp, 128>();
    else
        return R <= 32 ? simt::occupancy_pass2<Tp, 32>() : simt::occupancy_pass2<Tp, 64>();
}

template <typename Tp> int Simt<Tp>::chunk() { return simt::SB; }
template <typename Tp> int Simt<Tp>::oblock() { return simt::OB; }
template <typename Tp> int Simt<Tp>::rblock(int64_t R) { return simt::rblock_for<Tp>(R); }

template <typename Tp>
int Simt<Tp>::add_reg(const double* in, int64_t R, double reg, double* out, cudaStream_t st) {
    glue::k_add_reg<0><<<(unsigned)((R + 255) / 256), 256, 0, st>>>(in, R, reg, out);
    return simt::launch_status();
}

template <typename Tp>
int Simt<Tp>::raw_sums(const double* part, int64_t nparts, int64_t R, double* out,
                       cudaStream_t st) {
    if (R <= 1024)
        dna::launch_pdl(simt::k_colsum_small<0>, dim3((unsigned)R), dim3(256), 0, st, part,
                        (int)nparts, R, 0.0, out, false, nullptr);
    else
        simt::k_colsum_final<<<(unsigned)((R + 31) / 32), dim3(32, 32), 0, st>>>(
            part, (int)nparts, R, 0.0, out, false);
    return simt::launch_status();
}

namespace simt {
inline unsigned sp_grid(int64_t n) { return (unsigned)((n + sparse::WARPS - 1) / sparse::WARPS); }

// f(constant LPN) with the lanes per row of rank R (R <= 128)
template <class F>
int by_lanes(int64_t R, F&& f) {
    if (R <= 32) return f(std::integral_constant<int, 8>());
    if (R <= 64) return f(std::integral_constant<int, 16>());
    if (R <= 128) return f(std::integral_constant<int, 32>());
    return DNA_ERR_UNSUPPORTED;
}
}  // namespace simt

template <typename Tp>
int Simt<Tp>::sp_pass1(int64_t R, const SparseSegs& sg, const int32_t* idx, const Tp* val,
                       const Tp* Yr, const Tp* Xr, int64_t R4, Tp* Aseg, Tp* Bseg, bool with_b,
                       int* status, cudaStream_t st) {
    if (sg.n == 0) return DNA_OK;
    return simt::by_lanes(R, [&](auto lpn) {
        dna::launch_pdl(sparse::k_sp_pass1<Tp, decltype(lpn)::value>, dim3(simt::sp_grid(sg.n)),
                        dim3(sparse::WARPS * 32), 0, st, R4, sg, idx, val, Yr, Xr, Aseg, Bseg,
                        with_b, status);
        return simt::launch_status();
    });
}

template <typename Tp>
int Simt<Tp>::sp_cand(const View& v, const SparseSegs& sg, const Tp* Aseg, const Tp* Bseg,
                      const Tp* Xr, int64_t R4, const double* c, Tp* Xm, Tp* Xd, double eps,
                      double alpha, bool mu, const double* c0, Tp* c3, cudaStream_t st) {
    return simt::by_lanes(v.R, [&](auto lpn) {
        constexpr int LPN = decltype(lpn)::value;
        const unsigned grid = simt::sp_grid((v.O + 32 / LPN - 1) / (32 / LPN));
        auto k = mu ? sparse::k_sp_cand<Tp, LPN, true> : sparse::k_sp_cand<Tp, LPN, false>;
        dna::launch_pdl(k, grid, dim3(sparse::WARPS * 32), 0, st, v.O, v.R, R4, sg.sptr, Aseg,
                        Bseg, Xr, c, v.vsum, Xm, Xd, (Tp)eps, (Tp)alpha, c0, c3);
        return simt::launch_status();
    });
}

template <typename Tp>
int Simt<Tp>::sp_pass2(int64_t R, const SparseSegs& sg, const int32_t* idx, const Tp* val,
                       const Tp* Yr, const Tp* Xm, const Tp* Xd, int64_t R4, double* dseg,
                       cudaStream_t st) {
    if (sg.n == 0) return DNA_OK;
    return simt::by_lanes(R, [&](auto lpn) {
        dna::launch_pdl(sparse::k_sp_pass2<Tp, decltype(lpn)::value>, dim3(simt::sp_grid(sg.n)),
                        dim3(sparse::WARPS * 32), 0, st, R4, sg, idx, val, Yr, Xm, Xd, dseg);
        return simt::launch_status();
    });
}

template <typename Tp>
int Simt<Tp>::sp_select(const View& v, const SparseSegs& sg, const double* dseg, const Tp* Xm,
                        const Tp* Xd, int64_t R4, const Tp* c3, uint8_t* choice, double* dfin,
                        double* fpart, double reg, bool mu, int* status, cudaStream_t st) {
    return simt::by_lanes(v.R, [&](auto lpn) {
        constexpr int LPN = decltype(lpn)::value;
        auto k = mu ? sparse::k_sp_select<Tp, LPN, true> : sparse::k_sp_select<Tp, LPN, false>;
        dna::launch_pdl(k, dim3((unsigned)glue_parts(v.O)), dim3(sparse::WARPS * 32), 0, st, v,
                        R4, sg.sptr, dseg, Xm, Xd, c3, choice, dfin, fpart, reg, status);
        return simt::launch_status();
    });
}

template <typename Tp>
int Simt<Tp>::sp_kl(const View& v, const SparseSegs& sg, const int32_t* idx, const Tp* val,
                    const Tp* Yr, int64_t R4, const double* c0, double* dseg, double* part,
                    int* status, cudaStream_t st) {
    return simt::by_lanes(v.R, [&](auto lpn) {
        constexpr int LPN = decltype(lpn)::value;
        if (sg.n > 0) {
            sparse::k_sp_kl<Tp, LPN><<<simt::sp_grid(sg.n), sparse::WARPS * 32, 0, st>>>(
                v, R4, sg, idx, val, Yr, dseg);
            if (simt::launch_status()) return DNA_ERR_CUDA;
        }
        sparse::k_sp_reduce_kl<Tp, LPN><<<simt::sp_grid(v.O), sparse::WARPS * 32, 0, st>>>(
            v, sg.sptr, dseg, c0, part, status);
        return simt::launch_status();
    });
}

template <typename Tp>
int Simt<Tp>::pad_rows(const Tp* in, int64_t n, int64_t R, int64_t ld, Tp* out, cudaStream_t st) {
    const int64_t blocks = std::min<int64_t>((n * ld + 255) / 256, 152 * 16);
    dna::launch_pdl(sparse::k_pad_rows<Tp>, dim3((unsigned)blocks), dim3(256), 0, st, in, n, R,
                    ld, out);
    return simt::launch_status();
}

template <typename Tp>
int Simt<Tp>::transpose(const Tp* in, int64_t rows, int64_t cols, int64_t ld, Tp* out,
                        cudaStream_t st) {
    const dim3 grid((unsigned)((cols + 31) / 32), (unsigned)((ld + 31) / 32));
    dna::launch_pdl(sparse::k_transpose<Tp>, grid, dim3(32, 8), 0, st, in, rows, cols, ld, out);
    return simt::launch_status();
}

}  // namespace dna
