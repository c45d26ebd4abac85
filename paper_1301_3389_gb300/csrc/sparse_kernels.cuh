// Kernels of the sparse-V form (a DNA half-step that touches only the non-zeros of V).
//
// A half-step over the (s, o) view of Section 2 (H-step: o = column t, s = row n; W-step:
// o = row n, s = column t) needs z = (W H)_so only where v_so != 0: the ratios q = v/z and
// qbar = v/z^2 (steps 3, 10) are 0 elsewhere (the note after Algorithm 1), so A and B
// (eq. 7, 14) are sums over the non-zeros of the column, and so is the -v log z part of the
// candidates' costs (steps 9, 14).  The sum z part needs no zeros either:
// sum_s z_so = sum_r (sum_s y_sr) x_ro = sum_r c0_r x_ro with c0 the column sums of Y.
//
// Storage: the non-zeros of view column o are k in [ptr[o], ptr[o + 1]), at s = idx[k] with
// value val[k] (CSC of V for the H-step, CSR of V for the W-step).  Both factors are read as
// rows of R values padded with zeros to R4 = ceil(R / 4) 4 (W itself where R is a multiple
// of 4, else a padded copy; a transposed copy of H), and the candidates are rows [O][R4] too,
// so that every access of a lane is one 16-byte word of a contiguous row.
//
// Work is split into segments of at most SEG non-zeros of one view column (term rows of
// count data follow a Zipf law: one row can hold thousands of non-zeros), one warp per
// segment.  LPN = 8, 16 or 32 lanes (R <= 32, 64, 128) hold the four-value pieces of one row,
// so a warp works on 32 / LPN non-zeros (or view columns) at once: at R = 64 two rows per warp
// halve the shuffles and loads per non-zero against one row per warp with lane l holding
// r = l, l + 32.  What is left of the passes is the gather itself, 256 bytes per non-zero
// from L2 at 5 to 8 TB/s.  (A segment per lane group instead of per warp was no faster: 48, 65
// and 46, 61 us.)
// Each segment writes its partial sums [seg][R4], which the candidates kernel adds per
// column in order.  Sums over lanes run in a fixed order, so every result is
// bit-reproducible; the candidates' costs are summed across lanes and segments as three float32
// values each (sum3.cuh, no coarser than float64) because a float64 add costs 64 cycles per
// warp on this GPU.
// Measured at 36771 x 10212, 1.34 M non-zeros, R = 64 (H and W view, microseconds): pass 1
// 60, 73 -> 47, 66, pass 2 57, 70 -> 40, 54, sums of segments and candidates 20, 78 -> 6, 20,
// cost sums and selection 27, 81 -> 9, 15.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "dna_internal.h"
#include "simt_kernels.cuh"
#include "sum3.cuh"

namespace dna {
namespace sparse {

constexpr int WARPS = 8;   // warps per CTA
constexpr int U = 8;       // non-zeros per lane group whose loads are issued together
constexpr int SEG = SPARSE_SEG;

// Four consecutive values.
template <typename Tp>
struct Four {
    Tp v[4];
};
__device__ __forceinline__ Four<float> load4(const float* p) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    return {{t.x, t.y, t.z, t.w}};
}
__device__ __forceinline__ Four<double> load4(const double* p) {
    const double2 a = *reinterpret_cast<const double2*>(p);
    const double2 b = *reinterpret_cast<const double2*>(p + 2);
    return {{a.x, a.y, b.x, b.y}};
}
__device__ __forceinline__ void store4(float* p, const Four<float>& x) {
    *reinterpret_cast<float4*>(p) = make_float4(x.v[0], x.v[1], x.v[2], x.v[3]);
}
__device__ __forceinline__ void store4(double* p, const Four<double>& x) {
    *reinterpret_cast<double2*>(p) = make_double2(x.v[0], x.v[1]);
    *reinterpret_cast<double2*>(p + 2) = make_double2(x.v[2], x.v[3]);
}

// A sum over lanes or segments that loses nothing against float64: float64 itself, or for
// float32 values three of them (sum3.cuh).
template <typename Tp>
struct Sum;
template <>
struct Sum<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double t) { s += t; }
    __device__ __forceinline__ void add_product(double c, double, double, double x) { s += c * x; }
    // += what lane ^ m hands over
    __device__ __forceinline__ void add_from(const Sum& mine, int m) {
        s += __shfl_xor_sync(0xffffffffu, mine.s, m);
    }
    // += lane ^ m's sum
    __device__ __forceinline__ void add_lane(int m) { add_from(*this, m); }
    __device__ __forceinline__ void add_sum(const Sum& x) { s += x.s; }
    __device__ __forceinline__ bool past_range() const { return false; }
    __device__ __forceinline__ double value() const { return s; }
};
template <>
struct Sum<float> : Sum3 {
    __device__ __forceinline__ void add_sum(const Sum& x) { add(x.s, x.e, x.f); }
    __device__ __forceinline__ bool past_range() const { return large(s); }
    // the product of x with c0 + c1 + c2 (a float64 number cut in three)
    __device__ __forceinline__ void add_product(float c0, float c1, float c2, float x) {
        const float p = __fmul_rn(c0, x), q = __fmul_rn(c1, x);
        add(p);
        add_low(__fmaf_rn(c0, x, -p));
        add_low(q);
        f = __fadd_rn(f, __fmaf_rn(c2, x, __fmaf_rn(c1, x, -q)));
    }
    __device__ __forceinline__ void add_from(const Sum& mine, int m) {
        const float ts = __shfl_xor_sync(0xffffffffu, mine.s, m);
        const float te = __shfl_xor_sync(0xffffffffu, mine.e, m);
        const float tf = __shfl_xor_sync(0xffffffffu, mine.f, m);
        add(ts, te, tf);
    }
    __device__ __forceinline__ void add_lane(int m) {
        const float ts = __shfl_xor_sync(0xffffffffu, s, m);
        const float te = __shfl_xor_sync(0xffffffffu, e, m);
        const float tf = __shfl_xor_sync(0xffffffffu, f, m);
        // the same order on both sides of the exchange: the lower lane's sum first
        const bool up = (threadIdx.x & m) != 0;
        const float bs = up ? s : ts, be = up ? e : te, bf = up ? f : tf;
        s = up ? ts : s;
        e = up ? te : e;
        f = up ? tf : f;
        add(bs, be, bf);
    }
};
// the sums of x and y over groups of LPN lanes: x's in the lower half of the group, y's in the
// upper half (each half hands the other its own values first)
template <int LPN, typename Tp>
__device__ __forceinline__ Sum<Tp> group_add2(const Sum<Tp>& x, const Sum<Tp>& y) {
    const bool up = (threadIdx.x & (LPN / 2)) != 0;
    Sum<Tp> t = up ? y : x;
    t.add_from(up ? x : y, LPN / 2);
#pragma unroll
    for (int m = LPN / 4; m > 0; m >>= 1) t.add_lane(m);
    return t;
}
__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) x += __shfl_xor_sync(0xffffffffu, x, m);
    return x;
}
template <int LPN, typename Tp>
__device__ __forceinline__ Tp group_sum(Tp x) {
#pragma unroll
    for (int m = LPN / 2; m > 0; m >>= 1) x += __shfl_xor_sync(0xffffffffu, x, m);
    return x;
}

// The two cost sums of a segment, added over the warp's lanes and stored.  float32: two words of
// 16 bytes, each s, e, f and 0, or a float64 number, 0 and 1 where a lane's sum is near the end
// of float32's range (converting every segment's sums to float64 would cost ten float64
// instructions per warp and segment, a quarter of pass 2; the selection converts 32 columns
// at once).  float64: one word of 16 bytes.
__device__ __forceinline__ void store_costs(double* dseg, int64_t g, float m, float d) {
    const int lane = threadIdx.x & 31;
    float4* out = reinterpret_cast<float4*>(dseg) + 2 * g;
    if (__any_sync(0xffffffffu, Sum3::large(m) || Sum3::large(d))) {
        const double wm = warp_sum((double)m), wd = warp_sum((double)d);
        if (lane < 2) {
            const double t = lane ? wd : wm;
            out[lane] = make_float4(__int_as_float(__double2loint(t)),
                                    __int_as_float(__double2hiint(t)), 0.f, 1.f);
        }
        return;
    }
    // the lower half warp adds m, the upper half d
    const bool up = lane >= 16;
    Sum<float> x;
    x.add(up ? d : m);
    x.add(__shfl_xor_sync(0xffffffffu, up ? m : d, 16));
#pragma unroll
    for (int k = 8; k > 0; k >>= 1) x.add_lane(k);
    if (lane % 16 == 0) out[lane / 16] = make_float4(x.s, x.e, x.f, 0.f);
}
__device__ __forceinline__ void store_costs(double* dseg, int64_t g, double m, double d) {
    m = warp_sum(m);
    d = warp_sum(d);
    if (threadIdx.x % 32 == 0) reinterpret_cast<double2*>(dseg)[g] = make_double2(m, d);
}
__device__ __forceinline__ double word_value(const float4& t) {
    if (t.w != 0.f) return __hiloint2double(__float_as_int(t.y), __float_as_int(t.x));
    Sum3 x;
    x.s = t.x;
    x.e = t.y;
    x.f = t.z;
    return x.value();
}
// += the costs of the segments g0, g0 + step, ... < g1; whether a float64 number was among them
// (the sums are then of no use)
__device__ __forceinline__ bool add_costs(const double* dseg, int64_t g0, int64_t g1, int step,
                                          Sum<float>& m, Sum<float>& d) {
    const float4* w = reinterpret_cast<const float4*>(dseg);
    bool wide = false;
#pragma unroll 8
    for (int64_t g = g0; g < g1; g += step) {
        const float4 tm = w[2 * g], td = w[2 * g + 1];
        wide |= tm.w != 0.f || td.w != 0.f;
        m.add(tm.x, tm.y, tm.z);
        d.add(td.x, td.y, td.z);
    }
    return wide;
}
__device__ __forceinline__ bool add_costs(const double* dseg, int64_t g0, int64_t g1, int step,
                                          Sum<double>& m, Sum<double>& d) {
#pragma unroll 8
    for (int64_t g = g0; g < g1; g += step) {
        const double2 t = reinterpret_cast<const double2*>(dseg)[g];
        m.add(t.x);
        d.add(t.y);
    }
    return false;
}

// The non-zeros of a segment are read 32 at a time with one coalesced load (lane l holds
// the index and value of non-zero k + l) and handed to the whole warp by shuffles; the
// next 32 are loaded while the current ones are used, so each batch of non-zeros waits
// only for its gathered rows y(s, .).
template <typename Tp>
struct Chunk {
    int32_t s;
    Tp v;
};

template <typename Tp>
__device__ __forceinline__ Chunk<Tp> load_chunk(int64_t k, int64_t k1, int lane,
                                                const int32_t* __restrict__ idx,
                                                const Tp* __restrict__ val) {
    Chunk<Tp> c;
    const bool in = k + lane < k1;
    c.s = in ? idx[k + lane] : 0;
    c.v = in ? val[k + lane] : Tp(0);
    return c;
}

// Sums each of the NV per-lane values p[i] over groups of LPN lanes (NV a power of two, at
// most LPN) with a fixed reduce-scatter: at the step with xor mask m the lanes with bit m set
// keep the upper half of the remaining values and the others the lower half, each adding
// its partner's copy of the half it keeps; after log2(NV) steps a lane holds one value, index
// (lane % LPN) / (LPN / NV), and the remaining xor steps complete its sum.
template <int LPN, int NV, typename Tp>
__device__ __forceinline__ Tp scatter_sum(Tp (&p)[NV], int lane) {
    static_assert(NV >= 1 && NV <= LPN && (NV & (NV - 1)) == 0, "NV: a power of two <= LPN");
    int m = LPN / 2;
#pragma unroll
    for (int cnt = NV; cnt > 1; cnt >>= 1, m >>= 1) {
        const bool hi = (lane & m) != 0;
#pragma unroll
        for (int i = 0; i < cnt / 2; ++i) {
            const Tp keep = hi ? p[i + cnt / 2] : p[i];
            const Tp send = hi ? p[i] : p[i + cnt / 2];
            p[i] = keep + __shfl_xor_sync(0xffffffffu, send, m);
        }
    }
    Tp t = p[0];
#pragma unroll
    for (; m > 0; m >>= 1) t += __shfl_xor_sync(0xffffffffu, t, m);
    return t;
}

// Runs body(c, first, y) over the non-zeros [k0, k1) in batches of U per lane group: y[u] is
// the row of the non-zero whose index and value lane first + u holds in c (past the end: row
// 0 and value 0).
template <int LPN, typename Tp, class F>
__device__ __forceinline__ void for_nonzeros(int64_t k0, int64_t k1, int lane, int64_t R4,
                                             const int32_t* __restrict__ idx,
                                             const Tp* __restrict__ val,
                                             const Tp* __restrict__ Yr, F&& body) {
    constexpr int G = 32 / LPN;
    const int r = 4 * (lane % LPN);
    const bool in_row = r < R4;
    Chunk<Tp> cur = load_chunk<Tp>(k0, k1, lane, idx, val);
    for (int64_t k = k0; k < k1; k += 32) {
        const Chunk<Tp> nxt = load_chunk<Tp>(k + 32, k1, lane, idx, val);
        const int n = (int)(k1 - k < 32 ? k1 - k : 32);
        for (int base = 0; base < n; base += U * G) {
            const int first = base + U * (lane / LPN);
            Four<Tp> y[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t s = __shfl_sync(0xffffffffu, cur.s, first + u);
                if (in_row) y[u] = load4(Yr + s * R4 + r);
                else y[u] = Four<Tp>{{Tp(0), Tp(0), Tp(0), Tp(0)}};
            }
            body(cur, first, y);
        }
        cur = nxt;
    }
}

template <typename Tp>
__device__ __forceinline__ Tp dot4(const Four<Tp>& a, const Four<Tp>& b) {
    Tp t = a.v[0] * b.v[0];
#pragma unroll
    for (int i = 1; i < 4; ++i) t = fma(a.v[i], b.v[i], t);
    return t;
}

template <typename Tp>
__device__ __forceinline__ Four<Tp> row4(const Tp* __restrict__ M, int64_t row, int64_t R4, int r) {
    if (r < R4) return load4(M + row * R4 + r);
    return Four<Tp>{{Tp(0), Tp(0), Tp(0), Tp(0)}};
}

using Segs = SparseSegs;

// Pass 1 (Algorithm 1 steps 2-5 and 10 on the non-zeros of one segment): partial raw sums
// Aseg[g][r] = sum_k y(s_k, r) q_k and Bseg[g][r] = sum_k y(s_k, r)^2 qbar_k with q = v / z,
// qbar = q / z.  Sets STATUS_NONFINITE when z <= 0 (or is not a number) at a positive v.
template <typename Tp, int LPN>
__global__ void __launch_bounds__(WARPS * 32)
    k_sp_pass1(int64_t R4, Segs sg, const int32_t* __restrict__ idx, const Tp* __restrict__ val,
               const Tp* __restrict__ Yr, const Tp* __restrict__ Xr, Tp* __restrict__ Aseg,
               Tp* __restrict__ Bseg, bool with_b, int* __restrict__ status) {
    pdl_wait();
    constexpr int STEP = LPN / U;   // lanes that hold the same finished z
    const int lane = threadIdx.x & 31, sub = lane % LPN, lead = lane - sub, r = 4 * sub;
    const int64_t g = (int64_t)blockIdx.x * WARPS + (threadIdx.x >> 5);
    if (g >= sg.n) return;
    const int64_t k0 = sg.k0[g], k1 = sg.k1[g], col = sg.col[g];
    const Four<Tp> x = row4(Xr, col, R4, r);
    Four<Tp> a{{Tp(0), Tp(0), Tp(0), Tp(0)}}, b{{Tp(0), Tp(0), Tp(0), Tp(0)}};
    bool bad = false;
    for_nonzeros<LPN>(k0, k1, lane, R4, idx, val, Yr,
                      [&](const Chunk<Tp>& c, int first, const Four<Tp> (&y)[U]) {
        Tp p[U];
#pragma unroll
        for (int u = 0; u < U; ++u) p[u] = dot4(y[u], x);
        const Tp z = scatter_sum<LPN, U>(p, lane);            // z of non-zero sub / STEP
        const Tp vl = __shfl_sync(0xffffffffu, c.v, first + sub / STEP);
        Tp q = Tp(0), qb = Tp(0);
        if (vl > Tp(0)) {                                      // v = 0: q = qbar = 0
            if (z > Tp(0)) {
                const Tp rz = Tp(1) / z;                       // q = v / z, qbar = q / z
                q = vl * rz;
                qb = q * rz;
            } else {
                bad = true;
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const Tp qu = __shfl_sync(0xffffffffu, q, lead + u * STEP);
            const Tp qbu = __shfl_sync(0xffffffffu, qb, lead + u * STEP);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                a.v[i] = fma(y[u].v[i], qu, a.v[i]);
                b.v[i] = fma(y[u].v[i] * y[u].v[i], qbu, b.v[i]);
            }
        }
    });
#pragma unroll
    for (int m = LPN; m < 32; m <<= 1)   // the lane groups' shares of the segment
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            a.v[i] += __shfl_xor_sync(0xffffffffu, a.v[i], m);
            b.v[i] += __shfl_xor_sync(0xffffffffu, b.v[i], m);
        }
    if (lead == 0 && r < R4) {
        store4(Aseg + g * R4 + r, a);
        if (with_b) store4(Bseg + g * R4 + r, b);
    }
    bad = __any_sync(0xffffffffu, bad);
    if (bad && lane == 0) atomicOr(status, STATUS_NONFINITE);
}

// The candidates of view column o, a group of LPN lanes per column: A and B as the sums of
// the column's segments in order, then eq. 11 (Xm), eq. 15 / 17 and the eq. 10
// renormalisation (Xd), rows [O][R4] with zeros past R.  MU: Xm only.  c3 [3][4 LPN] receives the
// column sums c0 of Y, each as a sum of up to three values of the element type.
template <typename Tp, int LPN, bool MU>
__global__ void __launch_bounds__(WARPS * 32)
    k_sp_cand(int64_t O, int64_t R, int64_t R4, const int64_t* __restrict__ sptr,
              const Tp* __restrict__ Aseg, const Tp* __restrict__ Bseg,
              const Tp* __restrict__ Xr, const double* __restrict__ c,
              const double* __restrict__ vsum, Tp* __restrict__ Xm, Tp* __restrict__ Xd, Tp eps,
              Tp alpha, const double* __restrict__ c0, Tp* __restrict__ c3) {
    pdl_wait();
    pdl_next();
    if (!MU && blockIdx.x == 0)   // c0 as sums of three values, for the selection
        for (int k = threadIdx.x; k < 4 * LPN; k += WARPS * 32) {
            double t = k < R ? c0[k] : 0.0;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const Tp part = (Tp)t;
                c3[i * 4 * LPN + k] = part;
                t -= (double)part;
            }
        }
    __shared__ Tp cs[4 * LPN], ics[4 * LPN];
    for (int k = threadIdx.x; k < 4 * LPN; k += WARPS * 32) {
        cs[k] = k < R ? (Tp)c[k] : Tp(1);
        ics[k] = Tp(1) / cs[k];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, sub = lane % LPN, r = 4 * sub;
    const int64_t o =
        ((int64_t)blockIdx.x * WARPS + (threadIdx.x >> 5)) * (32 / LPN) + lane / LPN;
    const bool live = o < O;
    const bool in = live && r < R4;
    Four<Tp> a{{Tp(0), Tp(0), Tp(0), Tp(0)}}, b = a, x = a;
    if (in) {
        x = load4(Xr + o * R4 + r);
        const int64_t g1 = sptr[o + 1];
#pragma unroll 8
        for (int64_t g = sptr[o]; g < g1; ++g) {   // the longest columns have dozens
            const Four<Tp> ta = load4(Aseg + g * R4 + r);
#pragma unroll
            for (int i = 0; i < 4; ++i) a.v[i] += ta.v[i];
            if (!MU) {
                const Four<Tp> tb = load4(Bseg + g * R4 + r);
#pragma unroll
                for (int i = 0; i < 4; ++i) b.v[i] += tb.v[i];
            }
        }
    }
    Four<Tp> xm, xd;
    Tp den = Tp(0);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const Tp ic = ics[r + i], xr = x.v[i];
        if (MU) {
            xm.v[i] = xr * (a.v[i] / cs[r + i]);
            continue;
        }
        const Tp av = a.v[i] * ic - Tp(1), bv = b.v[i] * ic;   // eq. 7, 14
        xm.v[i] = xr * (a.v[i] * ic);      // eq. 11 as x (W^t q)_r / c_r (no cancellation)
        Tp d;
        if (av < Tp(0)) {                  // eq. 15, gain floored at eps
            const Tp xb = xr * bv;
            const Tp gn = simt::dev_div(xb, xb - av);
            d = xr * (gn > eps ? gn : eps);
        } else {                           // eq. 17, step capped at alpha x
            const Tp stp = bv > Tp(0) ? simt::dev_div(av, bv) : Tp(0);
            const Tp cap = alpha * xr;
            d = xr + (stp < cap ? stp : cap);
        }
        xd.v[i] = r + i < R ? d : Tp(0);
        den += cs[r + i] * xd.v[i];
    }
    if (in) store4(Xm + o * R4 + r, xm);
    if (MU) return;
    const Tp tot = group_sum<LPN>(den);    // eq. 10
    const Tp sc = live && tot > Tp(0) ? (Tp)vsum[o] / tot : Tp(1);
#pragma unroll
    for (int i = 0; i < 4; ++i) xd.v[i] *= sc;
    if (in) store4(Xd + o * R4 + r, xd);
}

// Pass 2 (steps 7-9, 12-14 on the non-zeros of one segment): the partial sums
// sum_{v>0} -v log z_MU and sum_{v>0} -v log z_DNA as the pair g of dseg.  A lane adds
// the terms of its non-zeros in the element type (at most SEG / U of them); the lanes' sums are
// added by store_costs.
template <typename Tp, int LPN>
__global__ void __launch_bounds__(WARPS * 32)
    k_sp_pass2(int64_t R4, Segs sg, const int32_t* __restrict__ idx, const Tp* __restrict__ val,
               const Tp* __restrict__ Yr, const Tp* __restrict__ Xm, const Tp* __restrict__ Xd,
               double* __restrict__ dseg) {
    pdl_wait();
    const int lane = threadIdx.x & 31, sub = lane % LPN, r = 4 * sub;
    const int64_t g = (int64_t)blockIdx.x * WARPS + (threadIdx.x >> 5);
    if (g >= sg.n) return;
    const int64_t k0 = sg.k0[g], k1 = sg.k1[g], col = sg.col[g];
    const Four<Tp> xm = row4(Xm, col, R4, r), xd = row4(Xd, col, R4, r);
    Tp lm_t = Tp(0), ld_t = Tp(0);
    for_nonzeros<LPN>(k0, k1, lane, R4, idx, val, Yr,
                      [&](const Chunk<Tp>& c, int first, const Four<Tp> (&y)[U]) {
        if constexpr (LPN >= 2 * U) {
            // a lane finishes one z: the MU z of non-zero u (values 0 .. U - 1) or the Newton
            // z (U .. 2U - 1); one lane of each value adds its term
            constexpr int STEP = LPN / (2 * U);
            Tp p[2 * U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                p[u] = dot4(y[u], xm);
                p[U + u] = dot4(y[u], xd);
            }
            const Tp z = scatter_sum<LPN, 2 * U>(p, lane);
            const int vi = sub / STEP;
            const Tp vl = __shfl_sync(0xffffffffu, c.v, first + vi % U);
            if (sub % STEP == 0 && vl > Tp(0)) {   // log of a non-positive z: NaN / -inf
                const Tp t = vl * log(z);
                if (vi < U) lm_t -= t; else ld_t -= t;
            }
        } else {   // as many lanes as non-zeros: a lane finishes both z of one
            static_assert(LPN == U || LPN >= 2 * U, "");
            Tp p[U], d[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                p[u] = dot4(y[u], xm);
                d[u] = dot4(y[u], xd);
            }
            const Tp zm = scatter_sum<LPN, U>(p, lane), zd = scatter_sum<LPN, U>(d, lane);
            const Tp vl = __shfl_sync(0xffffffffu, c.v, first + sub);
            if (vl > Tp(0)) {
                lm_t -= vl * log(zm);
                ld_t -= vl * log(zd);
            }
        }
    });
    store_costs(dseg, g, lm_t, ld_t);
}

// The cost of each candidate (the segments' sums in order, sum_s z = sum_r c0_r x(r, o), and
// reg sum_r x(r, o), the eq. 5 / eq. 4 penalty), the selection (Newton iff cheaper), the kept
// row into X, and fpart[blk][r] = sum over the CTA's 32 columns of the new x(r, o) (float64;
// the layout of k_select_fused).  MU: the row of Xm is kept.  A group of LPN lanes per column.
template <typename Tp, int LPN, bool MU>
__global__ void __launch_bounds__(WARPS * 32)
    k_sp_select(View v, int64_t R4, const int64_t* __restrict__ sptr,
                const double* __restrict__ dseg, const Tp* __restrict__ Xm,
                const Tp* __restrict__ Xd, const Tp* __restrict__ c3,
                uint8_t* __restrict__ choice, double* __restrict__ dfin,
                double* __restrict__ fpart, double reg, int* __restrict__ status) {
    pdl_wait();
    pdl_next();
    constexpr int G = 32 / LPN, NK = 4 / G;   // columns of a warp at once, rounds
    __shared__ Tp xs[4 * LPN][33];
    __shared__ Tp cc[3][4 * LPN];             // c0 as a sum of up to three values
    __shared__ Sum<Tp> sums[4][32];           // per column: sum z and sum x of both candidates
    __shared__ Sum<Tp> parts[WARPS][2][32];   // per column: shares of the segments' costs
    __shared__ int kept[32];
    const int64_t R = v.R, O = v.O, o0 = (int64_t)blockIdx.x * 32;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, sub = lane % LPN, r = 4 * sub;
    Four<Tp> x[NK], xd[NK];
    const Four<Tp> zero{{Tp(0), Tp(0), Tp(0), Tp(0)}};
#pragma unroll
    for (int k = 0; k < NK; ++k) {
        const int64_t o = o0 + 4 * w + k * G + lane / LPN;
        const bool in = o < O && r < R4;
        x[k] = in ? load4(Xm + o * R4 + r) : zero;
        if (!MU) xd[k] = in ? load4(Xd + o * R4 + r) : zero;
    }
    if (!MU) {
        for (int k = tid; k < 3 * 4 * LPN; k += WARPS * 32) cc[k / (4 * LPN)][k % (4 * LPN)] = c3[k];
        __syncthreads();
#pragma unroll
        for (int k = 0; k < NK; ++k) {
            Sum<Tp> zm, zd, pm, pd;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                zm.add_product(cc[0][r + i], cc[1][r + i], cc[2][r + i], x[k].v[i]);
                zd.add_product(cc[0][r + i], cc[1][r + i], cc[2][r + i], xd[k].v[i]);
            }
            zm = group_add2<LPN>(zm, zd);   // in the upper half of the group zd's sum
            if (reg != 0.0) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    pm.add(x[k].v[i]);
                    pd.add(xd[k].v[i]);
                }
                pm = group_add2<LPN>(pm, pd);
            }
            if (sub % (LPN / 2) == 0) {
                const int col = 4 * w + k * G + lane / LPN, which = sub != 0;
                sums[which][col] = zm;
                sums[2 + which][col] = pm;
            }
        }
        // lane = column: the segments' costs in order, or, where a column of the CTA has many of
        // them, warp w those at w, w + 8, ... and the eight sums in order
        const int64_t o = o0 + lane, g0 = o < O ? sptr[o] : 0, g1 = o < O ? sptr[o + 1] : 0;
        const bool many = __syncthreads_or(g1 - g0 > WARPS);
        Sum<Tp> lm, ld;
        bool wide = false;
        if (many || w == 0)
            wide = add_costs(dseg, g0 + (many ? w : 0), g1, many ? WARPS : 1, lm, ld);
        if (many) {
            parts[w][0][lane] = lm;
            parts[w][1][lane] = ld;
            wide = __syncthreads_or(wide);
            if (w == 0)
#pragma unroll
                for (int k = 1; k < WARPS; ++k) {
                    lm.add_sum(parts[k][0][lane]);
                    ld.add_sum(parts[k][1][lane]);
                }
        }
        if (w == 0) {   // float64 for 32 columns at once
            bool newton = false;
            if (o < O) {
                const Sum<Tp> zm = sums[0][lane], zd = sums[1][lane];
                lm.add_sum(zm);
                ld.add_sum(zd);
                double dm = lm.value(), dd = ld.value();
                if constexpr (sizeof(Tp) == 4)
                    if (wide || lm.past_range() || ld.past_range()) {
                        dm = dd = 0.0;
                        for (int64_t g = g0; g < g1; ++g) {
                            dm += word_value(reinterpret_cast<const float4*>(dseg)[2 * g]);
                            dd += word_value(reinterpret_cast<const float4*>(dseg)[2 * g + 1]);
                        }
                        dm += zm.value();
                        dd += zd.value();
                    }
                if (reg != 0.0) {
                    dm += reg * sums[2][lane].value();
                    dd += reg * sums[3][lane].value();
                }
                newton = dd < dm;
                choice[o] = newton ? 1 : 0;
                dfin[o] = dm;
                dfin[O + o] = dd;
                if (!isfinite(dm) || !isfinite(dd)) atomicOr(status, STATUS_NONFINITE);
            }
            kept[lane] = newton;
        }
        __syncthreads();
    }
    Tp* __restrict__ X = static_cast<Tp*>(v.X);
    const bool rows = v.xo != 1;   // X has contiguous rows of r
    const bool wide = R4 == R && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
#pragma unroll
    for (int k = 0; k < NK; ++k) {
        const int col = 4 * w + k * G + lane / LPN;
        const int64_t o = o0 + col;
        if (!MU && kept[col]) x[k] = xd[k];
#pragma unroll
        for (int i = 0; i < 4; ++i) xs[r + i][col] = x[k].v[i];
        if (rows && o < O && r < R) {
            if (wide) store4(X + o * v.xo + r, x[k]);
            else
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (r + i < R) X[o * v.xo + r + i] = x[k].v[i];
        }
    }
    __syncthreads();
    if (!rows && o0 + lane < O)
#pragma unroll 4
        for (int64_t q = w; q < R; q += WARPS) X[q * v.xr + o0 + lane] = xs[q][lane];
    for (int64_t q = tid; q < R; q += WARPS * 32) {
        Tp s = Tp(0);
#pragma unroll 8
        for (int i = 0; i < 32; ++i) s += xs[q][i];
        fpart[(int64_t)blockIdx.x * R + q] = (double)s;
    }
}

// d_KL (eq. 1) of the H view, per segment: sum over its non-zeros of v log(v / z) - v into
// dseg[g]: a lane's terms (at most SEG / U of them) in the element type, the lanes in float64.
template <typename Tp, int LPN>
__global__ void __launch_bounds__(WARPS * 32)
    k_sp_kl(View v, int64_t R4, Segs sg, const int32_t* __restrict__ idx,
            const Tp* __restrict__ val, const Tp* __restrict__ Yr, double* __restrict__ dseg) {
    constexpr int STEP = LPN / U;
    const int lane = threadIdx.x & 31, sub = lane % LPN, r = 4 * sub;
    const int64_t g = (int64_t)blockIdx.x * WARPS + (threadIdx.x >> 5);
    if (g >= sg.n) return;
    const int64_t k0 = sg.k0[g], k1 = sg.k1[g], col = sg.col[g];
    // the column of X, lane l reading r = l + 32 j
    __shared__ __align__(16) Tp xs[WARPS][4 * LPN];
    const Tp* __restrict__ X = static_cast<const Tp*>(v.X) + col * v.xo;
    Tp* xw = xs[threadIdx.x >> 5];
#pragma unroll
    for (int j = 0; j < LPN / 8; ++j) {
        const int q = lane + 32 * j;
        xw[q] = q < v.R ? X[q * v.xr] : Tp(0);
    }
    __syncwarp();
    const Four<Tp> x = load4(xw + r);
    Tp acc_t = Tp(0);   // the element type within the segment
    for_nonzeros<LPN>(k0, k1, lane, R4, idx, val, Yr,
                      [&](const Chunk<Tp>& c, int first, const Four<Tp> (&y)[U]) {
        Tp p[U];
#pragma unroll
        for (int u = 0; u < U; ++u) p[u] = dot4(y[u], x);
        const Tp z = scatter_sum<LPN, U>(p, lane);
        const Tp vl = __shfl_sync(0xffffffffu, c.v, first + sub / STEP);
        if (sub % STEP == 0 && vl > Tp(0)) acc_t += vl * log(vl / z) - vl;
    });
    const double t = warp_sum((double)acc_t);
    if (lane == 0) dseg[g] = t;
}

// Per column t of the H view: its segments' d_KL terms plus sum_n z_nt = sum_r c0_r h(r, t)
// into part[t].  A warp per column.
template <typename Tp, int LPN>
__global__ void __launch_bounds__(WARPS * 32)
    k_sp_reduce_kl(View v, const int64_t* __restrict__ sptr, const double* __restrict__ dseg,
                   const double* __restrict__ c0, double* __restrict__ part,
                   int* __restrict__ status) {
    constexpr int RPL = LPN / 8;   // values of r per lane
    const int lane = threadIdx.x & 31;
    const int64_t o = (int64_t)blockIdx.x * WARPS + (threadIdx.x >> 5);
    if (o >= v.O) return;
    const Tp* __restrict__ X = static_cast<const Tp*>(v.X) + o * v.xo;
    // all loads before the float64 chain (in a loop 34 us instead of 26 at T=20000 R=100)
    Tp x[RPL];
    double cr[RPL];
#pragma unroll
    for (int j = 0; j < RPL; ++j) {
        const int r = lane + 32 * j;
        x[j] = r < v.R ? X[r * v.xr] : Tp(0);
        cr[j] = r < v.R ? c0[r] : 0.0;
    }
    double zs = 0.0;
#pragma unroll
    for (int j = 0; j < RPL; ++j) zs += cr[j] * (double)x[j];
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) zs += __shfl_xor_sync(0xffffffffu, zs, m);
    if (lane == 0) {
        double acc = 0.0;
        for (int64_t g = sptr[o]; g < sptr[o + 1]; ++g) acc += dseg[g];
        const double d = acc + zs;
        part[o] = d;
        if (!isfinite(d)) atomicOr(status, STATUS_NONFINITE);
    }
}

// out[i][r] = in(i, r) for r < R, zeros up to ld: the rows of W (in[i * R + r]).
template <typename Tp>
__global__ void __launch_bounds__(256) k_pad_rows(const Tp* __restrict__ in, int64_t n, int64_t R,
                                                  int64_t ld, Tp* __restrict__ out) {
    pdl_wait();
    pdl_next();
    for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < n * ld;
         e += (int64_t)gridDim.x * 256) {
        const int64_t i = e / ld, r = e % ld;
        out[e] = r < R ? in[i * R + r] : Tp(0);
    }
}

// Rows of a factor stored along the other index: out[c * ld + r] = in[r * cols + c] (rows x
// cols row-major in), zeros for rows <= r < ld, through 32 x 32 shared-memory tiles so both
// sides stay coalesced.  CTA (32, 8).
template <typename Tp>
__global__ void __launch_bounds__(256) k_transpose(const Tp* __restrict__ in, int64_t rows,
                                                   int64_t cols, int64_t ld,
                                                   Tp* __restrict__ out) {
    pdl_wait();
    pdl_next();
    __shared__ Tp tile[32][33];
    const int64_t c0 = (int64_t)blockIdx.x * 32, r0 = (int64_t)blockIdx.y * 32;
    for (int i = threadIdx.y; i < 32; i += 8) {
        const int64_t r = r0 + i, c = c0 + threadIdx.x;
        tile[i][threadIdx.x] = (r < rows && c < cols) ? in[r * cols + c] : Tp(0);
    }
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += 8) {
        const int64_t c = c0 + i, r = r0 + threadIdx.x;
        if (c < cols && r < ld) out[c * ld + r] = tile[threadIdx.x][i];
    }
}

}  // namespace sparse
}  // namespace dna
