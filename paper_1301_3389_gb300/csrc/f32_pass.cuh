// The two O(NRT) passes of a half-step in float32 on the CUDA cores, ranks up to 128.
//
// The arithmetic is that of simt_kernels.cuh (pass 1: z = y x, q = v / z, qbar = v / z^2,
// A += y q, B += y^2 qbar; pass 2: the cost terms of the candidates' z).  These kernels are
// bound by the float32 FMA pipe, so everything is arranged around the packed instruction
// fma.rn.f32x2 (two FMAs per issue slot; a register-only loop reaches 65.7 TFLOP/s with
// it against 57.0 with scalar FMAs) and around few shared-memory wavefronts per FMA:
//  * A CTA of 256 threads owns 64 columns o and streams s in chunks of 64, two CTAs per SM,
//    so that one's loads and barriers hide behind the other's FMAs.
//  * Shared memory holds x as rows of o (Xs[r][o]) and y as rows of r (Ys[s][r]), padded so
//    that every access is free of bank conflicts.  In the z tile a thread owns 4 x 4 of
//    (s, o): pairs of o from one 16-byte load against y duplicated in registers, one
//    accumulator per z and r ascending.  In the A, B sums it pairs neighbouring r (8-byte
//    loads of Ys) against q duplicated in registers.
//  * A thread owns NR = RPT SG rows x 4 columns of A and B over 64 / SG of a chunk's s: the
//    rank is padded to a multiple of 16 only (R = 80 does not run as 128), and at small
//    ranks the SG groups of s keep 4 to 8 rows per thread instead of one.  With SG = 1 every
//    sum runs over s in ascending order within a split.
//  * Operands arrive by cp.async (zero-filled past the edges, 16 bytes wide where the rows
//    allow it), the next chunk's Y behind the present one's arithmetic where two Y tiles
//    fit; V goes by cp.async into the places of its own q.
// Measured against the kernels of simt_kernels.cuh (microseconds, H and W view, with the
// split plans of each): N=1024 T=11554 R=80 pass 1 304, 459 -> 152, 150 and pass 2 213, 368 ->
// 117, 119; N=4096 T=165 R=80 pass 1 203, 57 -> 23, 21; N=256 T=512 R=16 pass 1 24, 26 -> 6.6,
// 6.5.  At N=4096 T=16384 R=128 pass 1 runs at 45.5 TFLOP/s of algorithm, pass 2 at 40.8; the
// FMA pipe is busy 70 to 73 % of the time in pass 1, the rest is shared-memory bandwidth (two
// 16-byte loads per 8 packed FMAs in the z tile take as long as the FMAs) and the element-wise
// part.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "dna_internal.h"
#include "sum3.cuh"

namespace dna {
namespace f2 {

constexpr int NT = 256;   // threads per CTA
constexpr int OB = 64;    // o-block
constexpr int SB = 64;    // s-chunk
constexpr int LDX = 68;   // row length of the x tile [r][64 o]
constexpr int LDQ = 68;   // row length of the q, qbar tiles [s][64 o]

using u64 = unsigned long long;

__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
    u64 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 dup2(float x) {
    u64 d;
    asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(x));
    return d;
}
__device__ __forceinline__ float2 unpack2(u64 a) {
    float2 f;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(a));
    return f;
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
// copy 4 (16) bytes to shared memory asynchronously, zeros when !ok (nothing is read then)
__device__ __forceinline__ void cp4(uint32_t dst, const float* src, bool ok) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src),
                 "r"(ok ? 4 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp16(uint32_t dst, const float* src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src),
                 "r"(ok ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// y(s, r) at M[(s0 + i) si + r sr] into Ys[i][r], 64 rows of RB values (row length RB + 4),
// zero where s0 + i >= ns or r >= R.  si == 1 or sr == 1.
template <int RB>
__device__ __forceinline__ void load_y(float* sm, const float* __restrict__ M, int64_t si,
                                       int64_t sr, int64_t s0, int64_t ns, int64_t R) {
    constexpr int LDR = RB + 4;
    const int tid = threadIdx.x;
    const uint32_t base = smem_addr(sm);
    if (sr == 1) {
        if (((R | si) & 3) == 0 && (reinterpret_cast<uintptr_t>(M) & 15) == 0) {
#pragma unroll
            for (int k = 0; k < RB / 16; ++k) {
                const int e = tid + NT * k, i = e / (RB / 4), r = 4 * (e % (RB / 4));
                const bool ok = s0 + i < ns && r < R;
                cp16(base + 4u * (i * LDR + r), ok ? M + (s0 + i) * si + r : M, ok);
            }
        } else {
#pragma unroll 4
            for (int k = 0; k < RB / 4; ++k) {
                const int e = tid + NT * k, i = e / RB, r = e % RB;
                const bool ok = s0 + i < ns && r < R;
                cp4(base + 4u * (i * LDR + r), ok ? M + (s0 + i) * si + r : M, ok);
            }
        }
    } else {
        // a warp copies 8 rows x 4 values of r: whole 32-byte sectors of M, all 32 banks
        const int i = 8 * (tid >> 5) + (tid & 7), rl = (tid >> 3) & 3;
        const bool oki = s0 + i < ns;
        const float* p = M + s0 + i;
        const uint32_t dst = base + 4u * (i * LDR + rl);
#pragma unroll 4
        for (int k = 0; k < RB / 4; ++k) {
            const int r = 4 * k + rl;
            const bool ok = oki && r < R;
            cp4(dst + 16u * k, ok ? p + r * sr : M, ok);
        }
    }
}

// x(r, o) at M[r sr + (o0 + j) so] into Xs[r][j], RB rows of 64 values, zero where
// o0 + j >= no or r >= R.  so == 1 or sr == 1.
template <int RB>
__device__ __forceinline__ void load_x(float* sm, const float* __restrict__ M, int64_t sr,
                                       int64_t so, int64_t o0, int64_t no, int64_t R) {
    const int tid = threadIdx.x;
    const uint32_t base = smem_addr(sm);
    if (so == 1) {
        if (((no | sr) & 3) == 0 && (reinterpret_cast<uintptr_t>(M) & 15) == 0) {
#pragma unroll
            for (int k = 0; k < RB / 16; ++k) {
                const int e = tid + NT * k, r = e / 16, j = 4 * (e % 16);
                const bool ok = o0 + j < no && r < R;
                cp16(base + 4u * (r * LDX + j), ok ? M + r * sr + o0 + j : M, ok);
            }
        } else {
#pragma unroll 4
            for (int k = 0; k < RB / 4; ++k) {
                const int e = tid + NT * k, r = e / 64, j = e % 64;
                const bool ok = o0 + j < no && r < R;
                cp4(base + 4u * (r * LDX + j), ok ? M + r * sr + o0 + j : M, ok);
            }
        }
    } else {
        // a warp copies 8 values of r x 4 columns: whole sectors, all 32 banks
        const int rl = tid & 7, j0 = 8 * (tid >> 5) + ((tid >> 3) & 3);
#pragma unroll 4
        for (int k = 0; k < RB / 4; ++k) {
            const int r = 8 * (k >> 1) + rl, j = j0 + 4 * (k & 1);
            const bool ok = o0 + j < no && r < R;
            cp4(base + 4u * (r * LDX + j), ok ? M + (o0 + j) * so + r : M, ok);
        }
    }
}

// Where a thread works: rows s = sl + 16 i, columns o = 4 ol + j of the z tile.  A warp
// covers 4 x 8 of (sl, ol) with sl from lane bits 0 and 2, ol from bits 1, 3 and 4: a
// 16-byte shared load takes 4 cycles per warp, but 2.1 when lanes that differ in bit 0 (or
// in bit 1) read the same address (measured), which this order gives for both operands.
struct ZPos {
    int sl, ol;
};
__device__ __forceinline__ ZPos z_pos() {
    const int l = threadIdx.x & 31, w = threadIdx.x >> 5;
    return ZPos{(l & 1) + ((l >> 1) & 2) + 4 * (w >> 1),
                ((l >> 1) & 1) + ((l >> 2) & 6) + 8 * (w & 1)};
}

// z[k][i] = the four z(s, o) of row i (two pairs), summed over the first 4 nq values of r in
// ascending order, for the NC operands x_k in consecutive tiles of Xs.
template <int RB, int NC>
__device__ __forceinline__ void z_tile(const float* __restrict__ Ys, const float* __restrict__ Xs,
                                       ZPos p, int nq, u64 (&z)[NC][4][2]) {
    constexpr int LDR = RB + 4;
    const float* yp = Ys + p.sl * LDR;
    const float* xp = Xs + 4 * p.ol;
#pragma unroll
    for (int k = 0; k < NC; ++k)
#pragma unroll
        for (int i = 0; i < 4; ++i) { z[k][i][0] = 0ull; z[k][i][1] = 0ull; }
#pragma unroll 2
    for (int q = 0; q < nq; ++q) {
        float y[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 t = *reinterpret_cast<const float4*>(yp + 16 * i * LDR + 4 * q);
            y[i][0] = t.x; y[i][1] = t.y; y[i][2] = t.z; y[i][3] = t.w;
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            u64 d[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) d[i] = dup2(y[i][r]);
#pragma unroll
            for (int k = 0; k < NC; ++k) {
                const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(
                    xp + k * RB * LDX + (4 * q + r) * LDX);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    z[k][i][0] = fma2(d[i], x.x, z[k][i][0]);
                    z[k][i][1] = fma2(d[i], x.y, z[k][i][1]);
                }
            }
        }
    }
}

// Whether four neighbouring v(s, o .. o + 3), o a multiple of 4, are one aligned 16-byte word
// inside a row of V.
__device__ __forceinline__ bool v_wide(const View& v) {
    return ((v.vs | v.O) & 3) == 0 && (reinterpret_cast<uintptr_t>(v.V) & 15) == 0;
}
// v(s, o .. o + 3), zeros where s >= s_end or past the last column
__device__ __forceinline__ void load_v(const View& v, const float* __restrict__ V, bool wide,
                                       int64_t s, int64_t s_end, int64_t o, float (&x)[4]) {
    const float* p = V + s * v.vs + o;
    if (wide) {
        float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
        if (s < s_end && o < v.O) t = __ldg(reinterpret_cast<const float4*>(p));
        x[0] = t.x; x[1] = t.y; x[2] = t.z; x[3] = t.w;
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) x[j] = s < s_end && o + j < v.O ? __ldg(p + j) : 0.f;
    }
}

// Rank 16 RPT as SG groups of s x rows: each thread owns NR = RPT SG rows r in NP pairs
// (r = 2 rg + 2 NG p) and, when NR is odd, one single row (r = 2 NG NP + rg).
constexpr int s_groups(int rpt) { return rpt <= 2 ? 4 : rpt <= 4 ? 2 : 1; }

template <int RPT>
struct Tiles {
    static constexpr int RB = 16 * RPT, LDR = RB + 4;
    static constexpr int Y = SB * LDR, X = RB * LDX, Q = SB * LDQ;   // floats per tile
};

template <int RPT, bool WITH_B, int GROUPS>
struct Pass1 : Tiles<RPT> {
    using T = Tiles<RPT>;
    static constexpr int SG = GROUPS, NG = 16 / SG, NR = RPT * SG, NP = NR / 2, ODD = NR & 1;
    static constexpr int STAGES = RPT <= 6 ? 2 : 1;   // Y tiles: two CTAs fit an SM
    static constexpr int NQ = WITH_B ? 2 : 1;
    static constexpr size_t smem = sizeof(float) * (T::X + STAGES * T::Y + NQ * T::Q);
    // the s-groups' sums meet in shared memory at the end
    static_assert(sizeof(float) * (SG - 1) * (NT / SG) * NR * 4 * NQ <= smem, "");
};

// A and B sums of one (o-block, split of s): Apart / Bpart [splits][R][O].
template <int RPT, bool WITH_B, int GROUPS>
__device__ __forceinline__ void pass1_tile(const View& v, float* __restrict__ Apart,
                                           float* __restrict__ Bpart, int64_t s_per,
                                           int* __restrict__ status, int64_t tile_o,
                                           int64_t tile_s, float* sm) {
    using H = Pass1<RPT, WITH_B, GROUPS>;
    constexpr int LDR = H::LDR, NG = H::NG, NP = H::NP, ST = H::STAGES;
    float* Xs = sm;                       // [RB][LDX]
    float* Ys = Xs + H::X;                // [ST][64 s][LDR]
    float* Qs = Ys + ST * H::Y;           // [64 s][LDQ]: v, then q; then [64 s][LDQ]: qbar
    const float* __restrict__ V = static_cast<const float*>(v.V);
    const float* __restrict__ Y = static_cast<const float*>(v.Y);
    const int64_t o0 = tile_o * OB;
    const int64_t s_begin = tile_s * s_per, s_end = min(v.S, s_begin + s_per);
    const int nch = (int)((s_end - s_begin + SB - 1) / SB);
    const int nq = (int)((v.R + 3) / 4);
    const bool wide = v_wide(v);
    const ZPos zp = z_pos();
    const int rg = zp.sl % NG, sg = zp.sl / NG, og = zp.ol;

    u64 aA[NP > 0 ? NP : 1][4], aB[NP > 0 ? NP : 1][4];
    float sA[4], sB[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
        for (int p = 0; p < NP; ++p) { aA[p][j] = 0ull; aB[p][j] = 0ull; }
        sA[j] = 0.f;
        sB[j] = 0.f;
    }
    load_x<H::RB>(Xs, static_cast<const float*>(v.X), v.xr, v.xo, o0, v.O, v.R);
    load_y<H::RB>(Ys, Y, v.ys, v.yr, s_begin, v.S, v.R);
    cp_commit();
    int bad = 0;
    for (int c = 0; c < nch; ++c) {
        const int64_t s0 = s_begin + (int64_t)c * SB;
        float* Yc = Ys + (ST == 2 ? (c & 1) * H::Y : 0);
        if (ST == 1 && c > 0) {
            __syncthreads();   // every read of the previous chunk is done
            load_y<H::RB>(Ys, Y, v.ys, v.yr, s0, v.S, v.R);
            cp_commit();
        }
        if (ST == 2) {
            cp_wait<0>();
            __syncthreads();   // Y of this chunk is visible, the previous chunk's reads are done
        }
        {   // this thread's v, into the places of its q
            const int64_t o = o0 + 4 * zp.ol;
            const float* vp = V + (s0 + zp.sl) * v.vs + o;
            const uint32_t dst = smem_addr(Qs) + 4u * (zp.sl * LDQ + 4 * zp.ol);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const bool oks = s0 + zp.sl + 16 * i < s_end;
                if (wide) {
                    const bool ok = oks && o < v.O;
                    cp16(dst + 64u * i * LDQ, ok ? vp + 16 * i * v.vs : V, ok);
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const bool ok = oks && o + j < v.O;
                        cp4(dst + 64u * i * LDQ + 4u * j, ok ? vp + 16 * i * v.vs + j : V, ok);
                    }
                }
            }
            cp_commit();
        }
        if (ST == 2) {
            if (c + 1 < nch)
                load_y<H::RB>(Ys + (~c & 1) * H::Y, Y, v.ys, v.yr, s0 + SB, v.S, v.R);
            cp_commit();
        } else {
            cp_wait<1>();
            __syncthreads();
        }
        u64 z[1][4][2];
        z_tile<H::RB, 1>(Yc, Xs, zp, nq, z);
        cp_wait<(ST == 2 ? 1 : 0)>();   // this thread's own v
        // q = v / z, qbar = q / z, zero where v = 0 (note after Algorithm 1)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float* qp = Qs + (zp.sl + 16 * i) * LDQ + 4 * zp.ol;
            const float4 v4 = *reinterpret_cast<const float4*>(qp);
            const float vv[4] = {v4.x, v4.y, v4.z, v4.w};
            const float2 z0 = unpack2(z[0][i][0]), z1 = unpack2(z[0][i][1]);
            const float zz[4] = {z0.x, z0.y, z1.x, z1.y};
            float q[4], qb[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const bool pos = vv[j] > 0.f;
                bad |= (pos && !(zz[j] > 0.f)) ? 1 : 0;
                const float rz = __fdividef(1.f, zz[j]);
                q[j] = pos ? vv[j] * rz : 0.f;
                qb[j] = pos ? q[j] * rz : 0.f;
            }
            *reinterpret_cast<float4*>(qp) = make_float4(q[0], q[1], q[2], q[3]);
            if (WITH_B)
                *reinterpret_cast<float4*>(qp + H::Q) = make_float4(qb[0], qb[1], qb[2], qb[3]);
        }
        __syncthreads();
        {
            const float* yp = Yc + sg * (SB / H::SG) * LDR + 2 * rg;
            const float* qp = Qs + sg * (SB / H::SG) * LDQ + 4 * og;
            const float* yo = yp + 2 * NG * NP - rg;   // the single row
#pragma unroll 2
            for (int s = 0; s < SB / H::SG; ++s) {
                u64 y[NP > 0 ? NP : 1], d[4];
#pragma unroll
                for (int p = 0; p < NP; ++p)
                    y[p] = *reinterpret_cast<const u64*>(yp + s * LDR + 2 * NG * p);
                const float4 q4 = *reinterpret_cast<const float4*>(qp + s * LDQ);
                const float qq[4] = {q4.x, q4.y, q4.z, q4.w};
                float ys = 0.f;
                if (H::ODD) ys = yo[s * LDR];
#pragma unroll
                for (int j = 0; j < 4; ++j) d[j] = dup2(qq[j]);
#pragma unroll
                for (int p = 0; p < NP; ++p)
#pragma unroll
                    for (int j = 0; j < 4; ++j) aA[p][j] = fma2(y[p], d[j], aA[p][j]);
                if (H::ODD)
#pragma unroll
                    for (int j = 0; j < 4; ++j) sA[j] = fmaf(ys, qq[j], sA[j]);
                if (WITH_B) {
                    const float4 b4 = *reinterpret_cast<const float4*>(qp + H::Q + s * LDQ);
                    const float bb[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) d[j] = dup2(bb[j]);
#pragma unroll
                    for (int p = 0; p < NP; ++p) {
                        const u64 y2 = mul2(y[p], y[p]);
#pragma unroll
                        for (int j = 0; j < 4; ++j) aB[p][j] = fma2(y2, d[j], aB[p][j]);
                    }
                    if (H::ODD) {
                        const float y2 = ys * ys;
#pragma unroll
                        for (int j = 0; j < 4; ++j) sB[j] = fmaf(y2, bb[j], sB[j]);
                    }
                }
            }
        }
    }
    if (bad) atomicOr(status, STATUS_NONFINITE);

    // the sums of this thread as rows [NR][4] (A, then B)
    constexpr int NV = H::NR * 4 * H::NQ;
    float out[NV];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const float2 a = unpack2(aA[p][j]), b = unpack2(aB[p][j]);
            out[(2 * p) * 4 + j] = a.x;
            out[(2 * p + 1) * 4 + j] = a.y;
            if (WITH_B) {
                out[(H::NR + 2 * p) * 4 + j] = b.x;
                out[(H::NR + 2 * p + 1) * 4 + j] = b.y;
            }
        }
        if (H::ODD) {
            out[(H::NR - 1) * 4 + j] = sA[j];
            if (WITH_B) out[(2 * H::NR - 1) * 4 + j] = sB[j];
        }
    }
    if constexpr (H::SG > 1) {   // the s-groups' sums, added in order by group 0
        constexpr int TG = NT / H::SG;   // threads of one group
        const int tg = og * NG + rg;
        __syncthreads();
        if (sg > 0)
#pragma unroll
            for (int k = 0; k < NV; ++k) sm[((sg - 1) * NV + k) * TG + tg] = out[k];
        __syncthreads();
        if (sg == 0)
#pragma unroll
            for (int h = 0; h < H::SG - 1; ++h)
#pragma unroll
                for (int k = 0; k < NV; ++k) out[k] += sm[(h * NV + k) * TG + tg];
    }
    if (sg == 0) {
        const int64_t oc = o0 + 4 * og;
        const bool aligned = (v.O & 3) == 0;   // rows of A, B start on 16 bytes
#pragma unroll
        for (int m = 0; m < H::NQ; ++m) {
            float* P = (m ? Bpart : Apart) + tile_s * v.R * v.O + oc;
#pragma unroll
            for (int k = 0; k < H::NR; ++k) {
                const int r = k < 2 * NP ? 2 * rg + 2 * NG * (k / 2) + (k & 1) : 2 * NG * NP + rg;
                if (r >= v.R) continue;
                const float* x = out + (m * H::NR + k) * 4;
                if (aligned && oc < v.O)
                    *reinterpret_cast<float4*>(P + r * v.O) = make_float4(x[0], x[1], x[2], x[3]);
                else
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (oc + j < v.O) P[r * v.O + j] = x[j];
            }
        }
    }
}

// Chunks after which pass 2 moves its Sum3 to float64 (sum3.cuh: a run this long is at least as
// exact as float64 adds).
constexpr int SUM_RUN = 256;

template <int RPT, int NC>
struct Pass2 : Tiles<RPT> {
    using T = Tiles<RPT>;
    static constexpr int STAGES = NC == 1 || RPT <= 6 ? 2 : 1;
    static constexpr size_t tiles = sizeof(float) * (NC * T::X + STAGES * T::Y);
    static constexpr size_t red = 3 * sizeof(float) * 16 * NC * OB;
    static constexpr size_t smem = tiles > red ? tiles : red;
};

// This thread's cost sums of NC candidates over one (o-block, split of s), for the columns
// 4 ol + j: chunks of four terms in float32, added up in S (Sum3 or Sum64), which after
// every SUM_RUN chunks but the last ones is moved to acc.
// FULL = false: sum_{v>0} (-v log z) + sum z; FULL = true: the terms of eq. 1.
template <int RPT, int NC, bool FULL, class S>
__device__ __forceinline__ void pass2_sums(const View& v, const float* __restrict__ X0,
                                           const float* __restrict__ X1, int64_t xr, int64_t xo,
                                           int64_t o0, int64_t s_begin, int64_t s_end, int nch,
                                           int& bad, float* sm, S (&sums)[NC][4],
                                           double* __restrict__ acc) {
    using H = Pass2<RPT, NC>;
    constexpr int ST = H::STAGES;
    float* Xs = sm;                       // [NC][RB][LDX]
    float* Ys = Xs + NC * H::X;           // [ST][64 s][LDR]
    const float* __restrict__ V = static_cast<const float*>(v.V);
    const float* __restrict__ Y = static_cast<const float*>(v.Y);
    const int nq = (int)((v.R + 3) / 4);
    const bool wide = v_wide(v);
    const ZPos zp = z_pos();

    load_x<H::RB>(Xs, X0, xr, xo, o0, v.O, v.R);
    if (NC > 1) load_x<H::RB>(Xs + H::X, X1, xr, xo, o0, v.O, v.R);
    load_y<H::RB>(Ys, Y, v.ys, v.yr, s_begin, v.S, v.R);
    cp_commit();
    for (int c0 = 0; c0 < nch; c0 += SUM_RUN) {
        const int c1 = min(nch, c0 + SUM_RUN);
        for (int c = c0; c < c1; ++c) {
            const int64_t s0 = s_begin + (int64_t)c * SB;
            const float* Yc = Ys + (ST == 2 ? (c & 1) * H::Y : 0);
            if (ST == 1 && c > 0) {
                __syncthreads();
                load_y<H::RB>(Ys, Y, v.ys, v.yr, s0, v.S, v.R);
                cp_commit();
            }
            float vv[4][4];   // in flight behind the z FMAs
#pragma unroll
            for (int i = 0; i < 4; ++i)
                load_v(v, V, wide, s0 + zp.sl + 16 * i, s_end, o0 + 4 * zp.ol, vv[i]);
            cp_wait<0>();
            __syncthreads();
            if (ST == 2 && c + 1 < nch) {
                load_y<H::RB>(Ys + (~c & 1) * H::Y, Y, v.ys, v.yr, s0 + SB, v.S, v.R);
                cp_commit();
            }
            u64 z[NC][4][2];
            z_tile<H::RB, NC>(Yc, Xs, zp, nq, z);
#pragma unroll
            for (int k = 0; k < NC; ++k) {
                float run[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 z0 = unpack2(z[k][i][0]), z1 = unpack2(z[k][i][1]);
                    const float zr[4] = {z0.x, z0.y, z1.x, z1.y};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float zz = zr[j], x = vv[i][j];
                        const bool pos = x > 0.f;
                        bad |= (pos && !(zz > 0.f)) ? 1 : 0;
                        // branch-free: the v = 0 terms are discarded by the select
                        const float t = FULL ? (x * logf(x / zz) - x) : (-x * logf(zz));
                        run[j] += pos ? zz + t : zz;
                    }
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) sums[k][j].add(run[j]);
            }
        }
        if (c1 < nch)
#pragma unroll
            for (int k = 0; k < NC; ++k)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    acc[4 * k + j] = (c0 ? acc[4 * k + j] : 0.0) + sums[k][j].value();
                    sums[k][j] = S();
                }
    }
}

// The threads' float64 sums into red [16][NC][64].
template <int NC, class S>
__device__ __forceinline__ void put_sums(double* __restrict__ red, ZPos zp,
                                         const S (&sums)[NC][4], const double* __restrict__ acc,
                                         bool moved) {
#pragma unroll
    for (int k = 0; k < NC; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            red[(zp.sl * NC + k) * OB + 4 * zp.ol + j] =
                (moved ? acc[4 * k + j] : 0.0) + sums[k][j].value();
}

// The tile once more with float64 adds (rare: a call of its own, so that the usual path keeps
// its registers).
template <int RPT, int NC, bool FULL>
__device__ __noinline__ void pass2_again(const View& v, const float* X0, const float* X1,
                                         int64_t xr, int64_t xo, int64_t o0, int64_t s_begin,
                                         int64_t s_end, int nch, float* sm) {
    Sum64 sums[NC][4];
    double acc[4 * NC];
    int bad = 0;
    pass2_sums<RPT, NC, FULL>(v, X0, X1, xr, xo, o0, s_begin, s_end, nch, bad, sm, sums, acc);
    __syncthreads();
    put_sums<NC>(reinterpret_cast<double*>(sm), z_pos(), sums, acc, nch > SUM_RUN);
}

// Cost partials of NC candidates for one (o-block, split of s): dpart [splits][NC][O].  The
// sums run as Sum3 (a float64 add per chunk and column would take as long as the chunk's FMAs
// at small ranks; against pairs of float32, which are coarser than float64, iterations take
// 55.6 -> 55.5 us at N=256 T=512 R=16, 590 -> 596 at N=1024 T=11554 R=80, and 1156 -> 1175 for
// 48 problems in a group; a test of the range in the loop cost another 20).  Where a sum is
// infinite or has left float32's range, the tile is formed once more with float64 adds.
template <int RPT, int NC, bool FULL>
__device__ __forceinline__ void pass2_tile(const View& v, const float* __restrict__ X0,
                                           const float* __restrict__ X1, int64_t xr, int64_t xo,
                                           double* __restrict__ dpart, int64_t s_per,
                                           int* __restrict__ status, int64_t tile_o,
                                           int64_t tile_s, float* sm) {
    const int64_t o0 = tile_o * OB;
    const int64_t s_begin = tile_s * s_per, s_end = min(v.S, s_begin + s_per);
    const int nch = (int)((s_end - s_begin + SB - 1) / SB);
    const ZPos zp = z_pos();
    int bad = 0;
    double acc_mem[4 * NC];   // long splits only: kept out of the registers
    double* acc = acc_mem;
    asm volatile("" : "+l"(acc));
    Sum3 sums[NC][4];
    pass2_sums<RPT, NC, FULL>(v, X0, X1, xr, xo, o0, s_begin, s_end, nch, bad, sm, sums, acc);
    if (bad) atomicOr(status, STATUS_NONFINITE);

    // the 16 threads of each column, added in order
    const bool moved = nch > SUM_RUN;
    bool redo = false;
#pragma unroll
    for (int k = 0; k < NC; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            redo |= Sum3::large(sums[k][j].s) || isnan(sums[k][j].s);
            if (moved) redo |= !isfinite(acc[4 * k + j]);
        }
    const int tid = threadIdx.x, k = tid / OB, oo = tid % OB;
    double sum = 0.0;
    redo = __syncthreads_or(redo);   // and every read of the tiles is done
    if (redo || moved) {
        double* red = reinterpret_cast<double*>(sm);   // [16][NC][64]
        if (redo)
            pass2_again<RPT, NC, FULL>(v, X0, X1, xr, xo, o0, s_begin, s_end, nch, sm);
        else
            put_sums<NC>(red, zp, sums, acc, moved);
        __syncthreads();
        if (tid < NC * OB)
#pragma unroll
            for (int h = 0; h < 16; ++h) sum += red[(h * NC + k) * OB + oo];
    } else {   // as Sum3 too: one conversion to float64 per column
        constexpr int PL = 16 * NC * OB;   // [s, e, f][16][NC][64]
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const Sum3* x = sums[c];
            float* p = sm + (zp.sl * NC + c) * OB + 4 * zp.ol;
            *reinterpret_cast<float4*>(p) = make_float4(x[0].s, x[1].s, x[2].s, x[3].s);
            *reinterpret_cast<float4*>(p + PL) = make_float4(x[0].e, x[1].e, x[2].e, x[3].e);
            *reinterpret_cast<float4*>(p + 2 * PL) = make_float4(x[0].f, x[1].f, x[2].f, x[3].f);
        }
        __syncthreads();
        if (tid < NC * OB) {
            Sum3 t;
#pragma unroll
            for (int h = 0; h < 16; ++h) {
                const float* p = sm + (h * NC + k) * OB + oo;
                t.add(p[0], p[PL], p[2 * PL]);
            }
            sum = t.value();
        }
    }
    const int64_t o = o0 + oo;
    if (tid < NC * OB && o < v.O) dpart[(tile_s * NC + k) * v.O + o] = sum;
}

}  // namespace f2
}  // namespace dna
