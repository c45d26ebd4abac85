// The GEMM-shaped part of the adjoint of one H step in float32, ranks up to 128, with the
// step's dL/dW (both formulas and their derivation at k_adj_gemm and k_adj_wgrad in
// simt_kernels.cuh): from Abar = dL/dA, Bbar = dL/dB, per (s, o)
//   z = y x, P1 = y Abar, P2 = y^2 Bbar, q = v / z, qbar = q / z,
//   zbar = -qbar P1 - 2 (qbar / z) P2,
//   Vbar(s, o) += P1 / z + P2 / z^2 + vs_o,
//   Hpart(r, o) = sum_s y(s, r) zbar(s, o),
//   Wpart(s, r) = sum_o [Abar q + x zbar](s, o) + 2 y(s, r) sum_o [Bbar qbar](s, o).
// One kernel for both sums: the 64 x 64 tile of z, P1, P2 (6 R of the 14 R flop per element)
// is formed once, where separate kernels for H and W each formed it (20 R).  FMA-bound; the
// tiles, lane order and packed FMAs are those of f32_pass.cuh.  Six tiles ([r][o] of x,
// Abar, Bbar and [s][o] of q, qbar, zbar) and two of y leave room for one CTA per SM (two at
// ranks up to 32).  A CTA walks its group of o-blocks and, for each, its split of s: the H
// sums stay in registers over the split, the W sums of a chunk are added into the group's
// own partial in global memory, so that both partial counts stay small.
// Measured at N=1024 T=4096 R=64, per step: 103 us (H) + 207 us (W) in two kernels -> 134 us.
#include "f32_pass.cuh"

namespace dna {
namespace f2 {

template <int RPT>
struct Adj : Tiles<RPT> {
    using T = Tiles<RPT>;
    static constexpr int NP = RPT / 2, ODD = RPT & 1;
    static constexpr size_t smem = sizeof(float) * (3 * T::X + 2 * T::Y + 3 * T::Q);
};

template <int RPT, bool WITH_W>
__global__ void __launch_bounds__(NT, RPT <= 2 ? 2 : 1)
    k_adjoint_f2(View v, const float* __restrict__ Abar, const float* __restrict__ Bbar,
                 const double* __restrict__ vs, float* __restrict__ Hpart,
                 float* __restrict__ Vbar, int64_t ldvb, float* __restrict__ Wpart,
                 int64_t s_per, int64_t ob_per, int* __restrict__ status) {
    using H = Adj<RPT>;
    constexpr int RB = H::RB, LDR = H::LDR, NP = H::NP;
    extern __shared__ __align__(16) float smem_adj[];
    float* Xs = smem_adj;            // [RB][LDX] x, Abar, Bbar
    float* As = Xs + H::X;
    float* Bs = As + H::X;
    float* Ys = Bs + H::X;           // [2][64 s][LDR]
    float* Qs = Ys + 2 * H::Y;       // [64 s][LDQ] q, qbar, zbar
    float* Qb = Qs + H::Q;
    float* Zb = Qb + H::Q;
    const float* __restrict__ V = static_cast<const float*>(v.V);
    const float* __restrict__ Y = static_cast<const float*>(v.Y);
    const int64_t nob = (v.O + OB - 1) / OB;
    const int64_t ob0 = (int64_t)blockIdx.x * ob_per, ob1 = min(nob, ob0 + ob_per);
    const int64_t s_begin = (int64_t)blockIdx.y * s_per, s_end = min(v.S, s_begin + s_per);
    const int nch = (int)((s_end - s_begin + SB - 1) / SB);
    const int nq = (int)((v.R + 3) / 4);
    const bool wide = v_wide(v), wide_b = ((ldvb | v.O) & 3) == 0 &&
                                          (reinterpret_cast<uintptr_t>(Vbar) & 15) == 0;
    const ZPos zp = z_pos();
    int bad = 0;
    for (int64_t ob = ob0; ob < ob1; ++ob) {
        const int64_t o0 = ob * OB;
        load_x<RB>(Xs, static_cast<const float*>(v.X), v.xr, v.xo, o0, v.O, v.R);
        load_x<RB>(As, Abar, v.O, 1, o0, v.O, v.R);
        load_x<RB>(Bs, Bbar, v.O, 1, o0, v.O, v.R);
        load_y<RB>(Ys, Y, v.ys, v.yr, s_begin, v.S, v.R);
        cp_commit();
        u64 hp[NP > 0 ? NP : 1][4];
        float hs[4], vso[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
#pragma unroll
            for (int p = 0; p < NP; ++p) hp[p][j] = 0ull;
            hs[j] = 0.f;
            const int64_t o = o0 + 4 * zp.ol + j;
            vso[j] = o < v.O ? (float)vs[o] : 0.f;
        }
        for (int c = 0; c < nch; ++c) {
            const int64_t s0 = s_begin + (int64_t)c * SB;
            const float* Yc = Ys + (c & 1) * H::Y;
            float vv[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                load_v(v, V, wide, s0 + zp.sl + 16 * i, s_end, o0 + 4 * zp.ol, vv[i]);
            cp_wait<0>();
            __syncthreads();   // the operands are visible, the previous chunk's reads are done
            if (c + 1 < nch)
                load_y<RB>(Ys + (~c & 1) * H::Y, Y, v.ys, v.yr, s0 + SB, v.S, v.R);
            cp_commit();
            u64 z[4][2], p1[4][2], p2[4][2];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int h = 0; h < 2; ++h) { z[i][h] = 0ull; p1[i][h] = 0ull; p2[i][h] = 0ull; }
            {
                const float* yp = Yc + zp.sl * LDR;
                const float* xp = Xs + 4 * zp.ol;
#pragma unroll 1
                for (int q = 0; q < nq; ++q) {
                    float y[4][4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float4 t = *reinterpret_cast<const float4*>(yp + 16 * i * LDR + 4 * q);
                        y[i][0] = t.x; y[i][1] = t.y; y[i][2] = t.z; y[i][3] = t.w;
                    }
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const float* xr = xp + (4 * q + r) * LDX;
                        const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(xr);
                        const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(xr + H::X);
                        const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(xr + 2 * H::X);
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const u64 d = dup2(y[i][r]), d2 = mul2(d, d);
                            z[i][0] = fma2(d, x.x, z[i][0]);
                            z[i][1] = fma2(d, x.y, z[i][1]);
                            p1[i][0] = fma2(d, a.x, p1[i][0]);
                            p1[i][1] = fma2(d, a.y, p1[i][1]);
                            p2[i][0] = fma2(d2, b.x, p2[i][0]);
                            p2[i][1] = fma2(d2, b.y, p2[i][1]);
                        }
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int64_t s = s0 + zp.sl + 16 * i;
                float q[4], qb[4], zb[4], vb[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int64_t o = o0 + 4 * zp.ol + j;
                    const float2 zf = unpack2(z[i][j / 2]), f1 = unpack2(p1[i][j / 2]),
                                 f2 = unpack2(p2[i][j / 2]);
                    const float zz = j & 1 ? zf.y : zf.x, a = j & 1 ? f1.y : f1.x,
                                b = j & 1 ? f2.y : f2.x, x = vv[i][j];
                    const bool in = s < s_end && o < v.O, zpos = zz > 0.f;
                    bad |= in && x > 0.f && !zpos ? 1 : 0;
                    const float iz = zpos ? 1.f / zz : 0.f;
                    q[j] = x > 0.f ? x * iz : 0.f;
                    qb[j] = q[j] * iz;
                    zb[j] = -qb[j] * a - 2.f * qb[j] * iz * b;
                    vb[j] = vso[j] + a * iz + b * iz * iz;
                }
                if (Vbar && s < s_end) {
                    const int64_t o = o0 + 4 * zp.ol;
                    float* p = Vbar + s * ldvb + o;
                    if (wide_b) {
                        if (o < v.O) {
                            float4 t = *reinterpret_cast<float4*>(p);
                            t.x += vb[0]; t.y += vb[1]; t.z += vb[2]; t.w += vb[3];
                            *reinterpret_cast<float4*>(p) = t;
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (o + j < v.O) p[j] += vb[j];
                    }
                }
                const int at = (zp.sl + 16 * i) * LDQ + 4 * zp.ol;
                if (WITH_W) {
                    *reinterpret_cast<float4*>(Qs + at) = make_float4(q[0], q[1], q[2], q[3]);
                    *reinterpret_cast<float4*>(Qb + at) = make_float4(qb[0], qb[1], qb[2], qb[3]);
                }
                *reinterpret_cast<float4*>(Zb + at) = make_float4(zb[0], zb[1], zb[2], zb[3]);
            }
            __syncthreads();
            {   // Hpart(r, o) += sum_s y(s, r) zbar(s, o): r = 2 rg + 32 p, the single row last
                const int rg = zp.sl;
                const float* yp = Yc + 2 * rg;
                const float* yo = Yc + 32 * NP + rg;
                const float* qp = Zb + 4 * zp.ol;
#pragma unroll 4
                for (int s = 0; s < SB; ++s) {
                    const float4 q4 = *reinterpret_cast<const float4*>(qp + s * LDQ);
                    const float qq[4] = {q4.x, q4.y, q4.z, q4.w};
                    u64 d[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) d[j] = dup2(qq[j]);
#pragma unroll
                    for (int p = 0; p < NP; ++p) {
                        const u64 y = *reinterpret_cast<const u64*>(yp + s * LDR + 32 * p);
#pragma unroll
                        for (int j = 0; j < 4; ++j) hp[p][j] = fma2(y, d[j], hp[p][j]);
                    }
                    if (H::ODD) {
                        const float y = yo[s * LDR];
#pragma unroll
                        for (int j = 0; j < 4; ++j) hs[j] = fmaf(y, qq[j], hs[j]);
                    }
                }
            }
            if (WITH_W) {   // rows s = sl + 16 i, columns r = ol + 16 k; pairs of o
                u64 w1[4][RPT], w2[4][RPT];
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int k = 0; k < RPT; ++k) { w1[i][k] = 0ull; w2[i][k] = 0ull; }
                const float* qp = Qs + zp.sl * LDQ;
                const float* xp = Xs + zp.ol * LDX;
#pragma unroll 1
                for (int o = 0; o < OB; o += 4) {
                    ulonglong2 q[4], qb[4], zb[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float* p = qp + 16 * i * LDQ + o;
                        q[i] = *reinterpret_cast<const ulonglong2*>(p);
                        qb[i] = *reinterpret_cast<const ulonglong2*>(p + H::Q);
                        zb[i] = *reinterpret_cast<const ulonglong2*>(p + 2 * H::Q);
                    }
#pragma unroll
                    for (int k = 0; k < RPT; ++k) {
                        const float* p = xp + 16 * k * LDX + o;
                        const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(p);
                        const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(p + H::X);
                        const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(p + 2 * H::X);
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            w1[i][k] = fma2(q[i].x, a.x, fma2(zb[i].x, x.x, w1[i][k]));
                            w2[i][k] = fma2(qb[i].x, b.x, w2[i][k]);
                        }
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            w1[i][k] = fma2(q[i].y, a.y, fma2(zb[i].y, x.y, w1[i][k]));
                            w2[i][k] = fma2(qb[i].y, b.y, w2[i][k]);
                        }
                    }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int sl = zp.sl + 16 * i;
                    if (s0 + sl >= s_end) continue;
                    float* wp = Wpart + ((int64_t)blockIdx.x * v.S + s0 + sl) * v.R;
#pragma unroll
                    for (int k = 0; k < RPT; ++k) {
                        const int r = zp.ol + 16 * k;
                        if (r >= v.R) continue;
                        const float2 a = unpack2(w1[i][k]), b = unpack2(w2[i][k]);
                        const float t = a.x + a.y + 2.f * Yc[sl * LDR + r] * (b.x + b.y);
                        wp[r] = ob > ob0 ? wp[r] + t : t;
                    }
                }
            }
        }
        __syncthreads();   // the tiles are loaded again for the next o-block
        float* P = Hpart + (int64_t)blockIdx.y * v.R * v.O + o0 + 4 * zp.ol;
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
            const int r = k < 2 * NP ? 2 * zp.sl + 32 * (k / 2) + (k & 1) : 32 * NP + zp.sl;
            if (r >= v.R) continue;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float x = hs[j];
                if (k < 2 * NP) {
                    const float2 f = unpack2(hp[k < 2 * NP ? k / 2 : 0][j]);
                    x = k & 1 ? f.y : f.x;
                }
                if (o0 + 4 * zp.ol + j < v.O) P[r * v.O + j] = x;
            }
        }
    }
    if (bad) atomicOr(status, STATUS_NONFINITE);
}

template <int RPT, bool WITH_W>
static int launch(const View& v, const float* Abar, const float* Bbar, const double* vs,
                  float* Hpart, int splits, int64_t s_per, float* Vbar, int64_t ldvb,
                  float* Wpart, int groups, int64_t ob_per, int* status, cudaStream_t st) {
    auto k = k_adjoint_f2<RPT, WITH_W>;
    const size_t smem = Adj<RPT>::smem;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
        cudaSuccess)
        return DNA_ERR_CUDA;
    k<<<dim3((unsigned)groups, (unsigned)splits), NT, smem, st>>>(
        v, Abar, Bbar, vs, Hpart, Vbar, ldvb, Wpart, s_per, ob_per, status);
    return after_launch();
}

int adjoint(const View& v, const float* Abar, const float* Bbar, const double* vs, float* Hpart,
            int splits, int64_t s_per, float* Vbar, int64_t ldvb, float* Wpart, int groups,
            int64_t ob_per, int* status, cudaStream_t st) {
#define DNA_ADJ(N)                                                                             \
    case N:                                                                                    \
        return Wpart ? launch<N, true>(v, Abar, Bbar, vs, Hpart, splits, s_per, Vbar, ldvb,    \
                                       Wpart, groups, ob_per, status, st)                      \
                     : launch<N, false>(v, Abar, Bbar, vs, Hpart, splits, s_per, Vbar, ldvb,   \
                                        Wpart, groups, ob_per, status, st);
    switch ((v.R + 15) / 16) {
        DNA_ADJ(1) DNA_ADJ(2) DNA_ADJ(3) DNA_ADJ(4) DNA_ADJ(5) DNA_ADJ(6) DNA_ADJ(7) DNA_ADJ(8)
        default: return DNA_ERR_UNSUPPORTED;
    }
#undef DNA_ADJ
}

// Wbar(s, r) += sum over the groups of Wpart(s, r) + csum_r, both laid out like W (float64
// sums in ascending group order).
__global__ void __launch_bounds__(256)
    k_wgrad_add(const float* __restrict__ Wpart, int groups, const double* __restrict__ csum,
                int64_t n, int R, float* __restrict__ Wbar) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    double t = csum[i % R];
#pragma unroll 8
    for (int g = 0; g < groups; ++g) t += (double)Wpart[(int64_t)g * n + i];
    Wbar[i] = (float)((double)Wbar[i] + t);
}

int wgrad_add(const float* Wpart, int groups, const double* csum, int64_t S, int64_t R,
              float* Wbar, cudaStream_t st) {
    const int64_t n = S * R;
    k_wgrad_add<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(Wpart, groups, csum, n, (int)R, Wbar);
    return after_launch();
}

}  // namespace f2
}  // namespace dna
