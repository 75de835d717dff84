// k_data.cu -- the per-voxel data term (cost, gradient, Huber curvature), fused with the
// regulariser stencil, the NCG direction update and the monotonic line search.
//
// Per voxel j at field value w (Sec. II-III; see k_setup.cu for the pair factorisation):
//   Phi_j  = K_j + 4 sum_{m<n} |R_mn| sin^2(theta_mn / 2),  theta_mn = angle R_mn + w (t_m - t_n)
//   dPhi_j = 2 sum_{m<n} (t_m - t_n) |R_mn| sin(theta_mn)                         (Eq. 8)
//   d_j    = 2 sum_{m<n} (t_m - t_n)^2 sum_{c,d} |W_cm||W_dn| sinc(wrap(angle W_dn - angle W_cm
//                                                              + w (t_m - t_n)))  (Eq. 10-11)
// (the (n, m, d, c) term of every sum equals its (m, n, c, d) mirror, hence the factor 2),
// or, in the labelled FM_CURV_COMBINED variant and always for one coil,
//   d_j    = 2 sum_{m<n} (t_m - t_n)^2 |R_mn| sinc(wrap(theta_mn)).
// wrap() removes the nearest multiple of 2 pi ("mod pi" of Eq. 11 read as the wrap into
// [-pi, pi], Huber's optimal curvature for 1 - cos).
//
// FP32 mode evaluates the voxel arithmetic in float and sums in double; FP64 mode is double
// throughout.  Global sums are block partials reduced in a fixed order (bitwise
// reproducible).
#include <algorithm>
#include <type_traits>

#include "fm_internal.h"

namespace fm {

// ------------------------------------------------------------------ scalar helpers

__device__ __forceinline__ float wrap_angle(float t) {
    // nearest integer of t / (2 pi) by the 1.5 * 2^23 rounding constant (|t| < 2^21 here)
    const float k = fmaf(t, 0.159154943091895336f, 12582912.0f) - 12582912.0f;
    return fmaf(k, -6.28318530717958648f, t);
}
__device__ __forceinline__ double wrap_angle(double t) {
    return t - 6.283185307179586476925286766559 * rint(t * 0.15915494309189533576888376337251);
}

// sin(u)/u on the wrapped interval [-pi, pi] as a degree-5 polynomial in v = u^2: the
// discrete minimax fit derived by csrc/sinc_poly.py (truncation error 6.4e-8, 2.3e-7 overall
// in float Horner form, the level of float rounding of the weights).
__device__ __forceinline__ float sinc_wrapped(float u) {
    const float v = u * u;
    float p = -2.0676877099390367e-08f;
    p = fmaf(p, v, 2.708367901504971e-06f);
    p = fmaf(p, v, -0.00019817284191958606f);
    p = fmaf(p, v, 0.008332781493663788f);
    p = fmaf(p, v, -0.1666661947965622f);
    return fmaf(p, v, 0.9999999403953552f);
}
__device__ __forceinline__ double sinc_wrapped(double u) { return u == 0.0 ? 1.0 : sin(u) / u; }

// ------------------------------------------------------------------ FP32 literal curvature

// In FP32 mode (field-map model) the setup stores each coil weight's angle as a fixed-point
// fraction of a turn in the bits of the float slot: 2^32 is one turn, so a difference of two
// angles wraps into [-1/2, 1/2) turn by the integer subtraction's own wrap-around (Eq. 11's
// "mod pi" of the half angle).  The water-fat model and FP64 mode store radians.

__device__ __forceinline__ float fixed_to_radians(float bits) {
    return (float)__float_as_int(bits) * 1.4629180792671596e-09f;  // 2 pi / 2^32
}
// A stored coil angle in radians, for the general evaluator, which takes either storage.
template <typename T>
__device__ __forceinline__ T coil_angle(const DataArgs& a, T y) {
    if constexpr (sizeof(T) == 4) return a.wf ? y : fixed_to_radians(y);
    else return y;
}

// w (t_m - t_n) as a fixed-point angle (mod one turn) from dtt = (t_m - t_n) 2^32 / (2 pi):
// the float product split exactly into hi + lo, each rounded to an integer.
__device__ __forceinline__ unsigned phase_fixed(float w, float dtt) {
    const float hi = w * dtt, lo = fmaf(w, dtt, -hi);
    return (unsigned)(unsigned long long)__float2ll_rn(hi) + (unsigned)__float2int_rn(lo);
}

// The same reduced by turns in float before the conversion (the 64-bit conversion of phase_fixed
// runs on the narrow FP64 pipe).  Both hold to 2^24 turns, where lo leaves 32 bits; rintf and not the
// addition of 1.5 * 2^23, which finds whole turns below 2^22 only.
__device__ __forceinline__ unsigned phase_fixed_32(float w, float dtt) {
    const float hi = w * dtt, lo = fmaf(w, dtt, -hi);
    const float k = rintf(hi * 2.3283064365386963e-10f);  // whole turns
    return (unsigned)__float2int_rn(fmaf(k, -4294967296.0f, hi)) + (unsigned)__float2int_rn(lo);
}

// sin(2 pi x)/(2 pi x) for x in [-1/2, 1/2] turns as a degree-5 polynomial in x^2: the
// discrete minimax fit derived by csrc/sinc_poly.py (truncation error 6.1e-8, 2.1e-7 in
// float Horner form).
constexpr float kSincT0 = 0.9999999403953552f;
constexpr float kSincT1 = -6.579718589782715f;
constexpr float kSincT2 = 12.987038612365723f;
constexpr float kSincT3 = -12.193624496459961f;
constexpr float kSincT4 = 6.580165386199951f;
constexpr float kSincT5 = -1.9852460622787476f;

// The inner coil sum of Eq. 10 for one echo pair (m, n) in FP32, two coils d per
// instruction (the f32x2 forms of add, multiply and fused multiply-add, rounding each
// component as the scalar operation does):
//   sum_c |W_cm| sum_d |W_dn| sinc(wrap(angle W_dn + w (t_m - t_n) - angle W_cm)).
// Per term: the integer difference of the fixed-point angles (offset by half a turn, plus
// half of the 2^9 the shift drops, to round), one funnel shift that makes the float
// 1 + (difference + 1/2) in [1, 2) with 23 fraction bits, an exact subtraction of 1.5 that
// leaves the wrapped angle x in turns, and the degree-5 polynomial of sinc(2 pi x) in x^2
// (csrc/sinc_poly.py).  Even and odd d are summed apart, then added.
template <int NC>
__device__ __forceinline__ float coil_pair_sum_x2(const float2 (&Wm)[NC], const float2 (&Wn)[NC], unsigned ph) {
    static_assert(NC % 2 == 0, "two coils per instruction");
    constexpr int H = NC / 2;
    unsigned an[NC];
    float2 ad[H];
#pragma unroll
    for (int dd = 0; dd < NC; ++dd) an[dd] = (unsigned)__float_as_int(Wn[dd].y) + ph + 0x80000100u;
#pragma unroll
    for (int h = 0; h < H; ++h) ad[h] = make_float2(Wn[2 * h].x, Wn[2 * h + 1].x);
    const float2 c5 = make_float2(kSincT5, kSincT5), c4 = make_float2(kSincT4, kSincT4);
    const float2 c3 = make_float2(kSincT3, kSincT3), c2 = make_float2(kSincT2, kSincT2);
    const float2 c1 = make_float2(kSincT1, kSincT1), c0 = make_float2(kSincT0, kSincT0);
    const float2 mid = make_float2(-1.5f, -1.5f);
    float inner = 0;
#pragma unroll
    for (int cc = 0; cc < NC; ++cc) {
        const unsigned bm = (unsigned)__float_as_int(Wm[cc].y);
        float2 acc = make_float2(0.f, 0.f);
#pragma unroll
        for (int h = 0; h < H; ++h) {
            const float2 f = make_float2(__uint_as_float(__funnelshift_r(an[2 * h] - bm, 0x7Fu, 9)),
                                         __uint_as_float(__funnelshift_r(an[2 * h + 1] - bm, 0x7Fu, 9)));
            const float2 x = __fadd2_rn(f, mid);
            const float2 v = __fmul2_rn(x, x);
            float2 p = __ffma2_rn(c5, v, c4);
            p = __ffma2_rn(p, v, c3);
            p = __ffma2_rn(p, v, c2);
            p = __ffma2_rn(p, v, c1);
            p = __ffma2_rn(p, v, c0);
            acc = __ffma2_rn(ad[h], p, acc);
        }
        inner = fmaf(Wm[cc].x, acc.x + acc.y, inner);
    }
    return inner;
}

__device__ __forceinline__ void sin_cos(float x, float* s, float* c) { sincosf(x, s, c); }
__device__ __forceinline__ void sin_cos(double x, double* s, double* c) { sincos(x, s, c); }

// t_m - t_n of pair p in the voxel type
template <typename T>
__device__ __forceinline__ T pair_dt(const Pairs& pr, int p) {
    if constexpr (sizeof(T) == 4) return pr.dtf[p];
    else return pr.dt[p];
}

// ------------------------------------------------------------------ per-voxel data term

// Adds the data-term pieces of voxel j at field value w.  NC > 0: literal curvature over
// NC coils held in registers; NC == 0: literal curvature, runtime coil count; NC == 1:
// coil-combined curvature (exact for one coil).
template <typename T, int NC, bool COST, bool CURV>
__device__ __forceinline__ void eval_voxel(const DataArgs& a, long long j /* compact index */, T w, T& cost,
                                           T& grad, T& curv) {
    using T2 = typename V2<T>::t;
    const long long nv = a.geo.nv;
    const T2* pairs = (const T2*)a.pairs;
    const T2* coils = (const T2*)a.coils;
    T c_acc = 0, g_acc = 0, d_acc = 0;
    if constexpr (NC == 1) {
        // the pair weights are all there is to load: kB at a time, before their arithmetic (one at
        // a time the loop waits for each; six echoes, 15 pairs, 192 x 192 x 64 voxels, line search: 235 -> 206 us)
        constexpr int kB = 5;
        for (int p0 = 0; p0 < a.pr.P; p0 += kB) {
            T2 R[kB];
#pragma unroll
            for (int i = 0; i < kB; ++i)
                if (p0 + i < a.pr.P) R[i] = pairs[(size_t)(p0 + i) * nv + j];
#pragma unroll
            for (int i = 0; i < kB; ++i) {
                if (p0 + i >= a.pr.P) break;
                const T dt = pair_dt<T>(a.pr, p0 + i);
                const T th = R[i].y + w * dt;
                T s, c;
                sin_cos(th * T(0.5), &s, &c);
                if (COST) c_acc += R[i].x * (s * s);
                g_acc += dt * R[i].x * (s * c);
                if (CURV) d_acc += dt * dt * R[i].x * sinc_wrapped(wrap_angle(th));
            }
        }
        cost = T(4) * c_acc;
        grad = T(4) * g_acc;
        curv = T(2) * d_acc;
        return;
    }
    for (int p = 0; p < a.pr.P; ++p) {
        const T dt = pair_dt<T>(a.pr, p);
        const T2 R = pairs[(size_t)p * nv + j];
        const T th = R.y + w * dt;
        T s, c;
        sin_cos(th * T(0.5), &s, &c);
        if (COST) c_acc += R.x * (s * s);
        g_acc += dt * R.x * (s * c);
        if (CURV) {
            if (NC > 1) {
                const int m = a.pr.m[p], n = a.pr.n[p];
                T psi[NC > 1 ? NC : 1], ad[NC > 1 ? NC : 1];
#pragma unroll
                for (int dd = 0; dd < NC; ++dd) {
                    const T2 q = coils[((size_t)n * NC + dd) * nv + j];
                    ad[dd] = q.x;
                    psi[dd] = q.y + w * dt;
                }
                T inner = 0;
#pragma unroll
                for (int cc = 0; cc < NC; ++cc) {
                    const T2 q = coils[((size_t)m * NC + cc) * nv + j];
                    T acc = 0;
#pragma unroll
                    for (int dd = 0; dd < NC; ++dd) acc += ad[dd] * sinc_wrapped(wrap_angle(psi[dd] - q.y));
                    inner += q.x * acc;
                }
                d_acc += dt * dt * inner;
            } else {
                // runtime coil count (FP64), and the water-fat model, whose angle r_cdmn carries the
                // phase of Gamma_mn and |r_cdmn| the factor L |Gamma_mn| (0 and 1 otherwise)
                const int m = a.pr.m[p], n = a.pr.n[p], nc = a.nc;
                const T gph = (T)a.pr.gph[p];
                T inner = 0;
                for (int cc = 0; cc < nc; ++cc) {
                    const T2 q = coils[((size_t)m * nc + cc) * nv + j];
                    T acc = 0;
                    for (int dd = 0; dd < nc; ++dd) {
                        const T2 r = coils[((size_t)n * nc + dd) * nv + j];
                        acc += r.x * sinc_wrapped(wrap_angle(coil_angle(a, r.y) + w * dt + gph - coil_angle(a, q.y)));
                    }
                    inner += q.x * acc;
                }
                d_acc += dt * dt * (T)a.pr.gmag[p] * inner;
            }
        }
    }
    cost = T(4) * c_acc;
    grad = T(4) * g_acc;
    curv = T(2) * d_acc;
}

// Same as eval_voxel for a compile-time echo count L: the pair loop is unrolled and every
// pair and coil value of the voxel is loaded before the arithmetic starts -- by load(), which
// needs the compact index alone, so that a kernel can put it before its own gathers.
template <typename T, int NC, int L, bool CURV>
struct VoxelData {
    using T2 = typename V2<T>::t;
    static constexpr int P = L * (L - 1) / 2, NCL = (CURV && NC > 1) ? NC : 1;
    T2 R[P];
    T2 W[L][NCL];
    __device__ __forceinline__ void load(const DataArgs& a, long long j /* compact index */) {
        const long long nv = a.geo.nv;
        const T2* pairs = (const T2*)a.pairs;
        const T2* coils = (const T2*)a.coils;
#pragma unroll
        for (int p = 0; p < P; ++p) R[p] = pairs[(size_t)p * nv + j];
        if (CURV && NC > 1) {
#pragma unroll
            for (int m = 0; m < L; ++m)
#pragma unroll
                for (int c = 0; c < NCL; ++c) W[m][c] = coils[((size_t)m * NC + c) * nv + j];
        }
    }
    template <bool COST>
    __device__ __forceinline__ void eval(const DataArgs& a, T w, T& cost, T& grad, T& curv) const;
};

template <typename T, int NC, int L, bool CURV>
template <bool COST>
__device__ __forceinline__ void VoxelData<T, NC, L, CURV>::eval(const DataArgs& a, T w, T& cost, T& grad, T& curv) const {
    T c_acc = 0, g_acc = 0, d_acc = 0;
    int p = 0;
#pragma unroll
    for (int m = 0; m < L; ++m) {
#pragma unroll
        for (int n = m + 1; n < L; ++n, ++p) {
            const T dt = pair_dt<T>(a.pr, p);
            const T th = R[p].y + w * dt;
            T s, c;
            sin_cos(th * T(0.5), &s, &c);
            if (COST) c_acc += R[p].x * (s * s);
            g_acc += dt * R[p].x * (s * c);
            if (CURV) {
                if constexpr (NC == 1) {
                    d_acc += dt * dt * R[p].x * sinc_wrapped(wrap_angle(th));
                } else if constexpr (sizeof(T) == 4 && NCL % 2 == 0) {
                    d_acc += dt * dt * coil_pair_sum_x2<NCL>(W[m], W[n], phase_fixed(w, a.pr.dtt[p]));
                } else {
                    T psi[NCL];
#pragma unroll
                    for (int dd = 0; dd < NCL; ++dd) psi[dd] = W[n][dd].y + w * dt;
                    T inner = 0;
#pragma unroll
                    for (int cc = 0; cc < NCL; ++cc) {
                        T acc = 0;
#pragma unroll
                        for (int dd = 0; dd < NCL; ++dd)
                            acc += W[n][dd].x * sinc_wrapped(wrap_angle(psi[dd] - W[m][cc].y));
                        inner += W[m][cc].x * acc;
                    }
                    d_acc += dt * dt * inner;
                }
            }
        }
    }
    cost = T(4) * c_acc;
    grad = T(4) * g_acc;
    curv = T(2) * d_acc;
}

template <typename T, int NC, int L, bool COST, bool CURV>
__device__ __forceinline__ void eval_fixed(const DataArgs& a, long long j, T w, T& cost, T& grad, T& curv) {
    VoxelData<T, NC, L, CURV> v;
    v.load(a, j);
    v.template eval<COST>(a, w, cost, grad, curv);
}

// FP32 literal curvature of up to NR coils (two coils per instruction, so NR is even) and any
// echo count: a pair's coil weights in registers, coils past a.nc counting as |W| = 0.  Bound by
// FP32 issue at 6 slots per term of NR^2; the runtime-count form it replaces took 11 to 15 per
// term.  133 x 117 x 45 voxels, four coils and echoes: line search 163 -> 129 us, gradient 32 -> 28
// (96 and 30 in the present build).
template <int NR, bool COST, bool CURV>
__device__ __forceinline__ void eval_padded(const DataArgs& a, long long j, float w, float& cost, float& grad,
                                            float& curv) {
    const size_t nv = (size_t)a.geo.nv;
    const float2* pairs = (const float2*)a.pairs + j;
    const float2* coils = (const float2*)a.coils + j;
    const int nc = a.nc, L = a.L;
    auto load = [&](float2 (&W)[NR], int m) {
#pragma unroll
        for (int c = 0; c < NR; ++c) W[c] = c < nc ? coils[(size_t)(m * nc + c) * nv] : make_float2(0.f, 0.f);
    };
    float c_acc = 0, g_acc = 0, d_acc = 0;
    int p = 0;
    for (int m = 0; m + 1 < L; ++m) {
        float2 Wm[NR];
        if (CURV) load(Wm, m);
        for (int n = m + 1; n < L; ++n, ++p) {
            float2 Wn[NR];
            if (CURV) load(Wn, n);
            const float dt = a.pr.dtf[p];
            const float2 R = pairs[(size_t)p * nv];
            float s, c;
            sin_cos((R.y + w * dt) * 0.5f, &s, &c);
            if (COST) c_acc += R.x * (s * s);
            g_acc += dt * R.x * (s * c);
            if (CURV) d_acc += dt * dt * coil_pair_sum_x2<NR>(Wm, Wn, phase_fixed_32(w, a.pr.dtt[p]));
        }
    }
    cost = 4.f * c_acc;
    grad = 4.f * g_acc;
    curv = 2.f * d_acc;
}

// ------------------------------------------------------------------ voxels shared by lanes

// FP32 literal curvature of more than eight coils, any echo count: SP lanes share a voxel, eight or
// one (slice_lanes).  Lane slice sl takes the rows c = sl, sl + SP, .. of every pair's sum over (c, d),
// and the pairs sl, sl + SP, .. of the cost and gradient; the slices' results add up to the voxel's.
//
// Bound by FP32 issue: a pair has N_c^2 terms of about 6 slots.  A lane holds eight d in registers for
// all of its rows, two terms per instruction as in coil_pair_sum_x2 (with one coil load per term and no
// reuse, 11 to 15 slots a term).  One lane per voxel leaves the chip idle where coils are many and
// voxels few: 74 x 74 x 10 voxels with 32 coils are 14,000 mask voxels for 152 SMs, 3072 terms each, and
// their line search took 630 us, with eight lanes per voxel 205 (gradient 108, 47).  The lanes of a slice
// are neighbouring voxels, so that a load fetches whole 32-byte sectors of each coil's plane.  Up to
// eight coils are eval_padded's, which holds both sides of a pair in registers.

// sum over the rows c = sl, sl + SP, .. of |W_cm| sum_{d < DB} |W_dn| sinc(..), entries past the last
// of nd coils counting as |W_dn| = 0.
template <int SP, int DB>
__device__ __forceinline__ float slice_block(const float2* Wm, const float2* Wn, size_t nv, int nc, int sl, int nd,
                                             unsigned ph) {
    unsigned an[DB];
    float2 ad[DB / 2];
#pragma unroll
    for (int i = 0; i < DB; ++i, Wn += nv) {
        const float2 r = i < nd ? *Wn : make_float2(0.f, 0.f);
        an[i] = (unsigned)__float_as_int(r.y) + ph + 0x80000100u;
        if (i & 1) ad[i / 2].y = r.x;
        else ad[i / 2].x = r.x;
    }
    const float2 c5 = make_float2(kSincT5, kSincT5), c4 = make_float2(kSincT4, kSincT4);
    const float2 c3 = make_float2(kSincT3, kSincT3), c2 = make_float2(kSincT2, kSincT2);
    const float2 c1 = make_float2(kSincT1, kSincT1), c0 = make_float2(kSincT0, kSincT0);
    const float2 mid = make_float2(-1.5f, -1.5f);
    float inner = 0;
    Wm += (size_t)sl * nv;
#pragma unroll 2
    for (int c = sl; c < nc; c += SP, Wm += SP * nv) {
        const float2 q = *Wm;
        const unsigned bm = (unsigned)__float_as_int(q.y);
        float2 acc = make_float2(0.f, 0.f);
#pragma unroll
        for (int h = 0; h < DB / 2; ++h) {
            const float2 f = make_float2(__uint_as_float(__funnelshift_r(an[2 * h] - bm, 0x7Fu, 9)),
                                         __uint_as_float(__funnelshift_r(an[2 * h + 1] - bm, 0x7Fu, 9)));
            const float2 x = __fadd2_rn(f, mid);
            const float2 v = __fmul2_rn(x, x);
            float2 p = __ffma2_rn(c5, v, c4);
            p = __ffma2_rn(p, v, c3);
            p = __ffma2_rn(p, v, c2);
            p = __ffma2_rn(p, v, c1);
            p = __ffma2_rn(p, v, c0);
            acc = __ffma2_rn(ad[h], p, acc);
        }
        inner = fmaf(q.x, acc.x + acc.y, inner);
    }
    return inner;
}

// This slice's share of voxel k's cost, gradient and curvature at field value w.
template <int SP, bool COST>
__device__ __forceinline__ void eval_slice(const DataArgs& a, long long k, int sl, float w, float& cost, float& grad,
                                           float& curv) {
    const size_t nv = (size_t)a.geo.nv;
    const float2* pairs = (const float2*)a.pairs + k;
    const float2* coils = (const float2*)a.coils + k;
    const int nc = a.nc, P = a.pr.P;
    float c_acc = 0, g_acc = 0, d_acc = 0;
    for (int p = sl; p < P; p += SP) {
        const float dt = a.pr.dtf[p];
        const float2 R = pairs[(size_t)p * nv];
        float s, c;
        sin_cos((R.y + w * dt) * 0.5f, &s, &c);
        if (COST) c_acc += R.x * (s * s);
        g_acc += dt * R.x * (s * c);
    }
    for (int p = 0; p < P; ++p) {
        const float dt = a.pr.dtf[p];
        const unsigned ph = phase_fixed_32(w, a.pr.dtt[p]);
        const float2 *Wm = coils + (size_t)a.pr.m[p] * nc * nv, *Wn = coils + (size_t)a.pr.n[p] * nc * nv;
        float inner = 0;
        int d0 = 0;
        for (; d0 + 4 < nc; d0 += 8, Wn += 8 * nv) inner += slice_block<SP, 8>(Wm, Wn, nv, nc, sl, nc - d0, ph);
        if (d0 < nc) inner += slice_block<SP, 4>(Wm, Wn, nv, nc, sl, nc - d0, ph);
        d_acc += dt * dt * inner;
    }
    cost = 4.f * c_acc;
    grad = 4.f * g_acc;
    curv = 2.f * d_acc;
}

// The sum of v over the SP lanes of a voxel (lane = slice * (32 / SP) + voxel), in all of them.
template <int SP>
__device__ __forceinline__ float slice_sum(float v) {
#pragma unroll
    for (int o = 32 / SP; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Lanes that share a voxel of a mask of nm voxels: kShared while the chip holds them in few rounds (9728
// voxels with eight lanes each, two blocks per SM), else one, as a lane of its own keeps a voxel's rows
// even and its loads whole (eight lanes have 16 rows' time for nine coils).  The more coils, the later:
// line search / gradient in us with one and with eight lanes, three echoes, 9216 voxels: 9 coils 74 / 18
// and 55 / 16, 32 coils 390 / 53 and 96 / 25; 20,480: 9 coils 76 / 20 and 95 / 31, 16 coils 127 / 26 and
// 92 / 28, 32 coils 392 / 57 and 210 / 47; 82,944: 16 coils 227 / 45 and 212 / 63, 32 coils 759 / 127 and
// 561 / 133; 393,216: 9 coils 332 / 77 and 1005 / 315.  With two echoes the pair's work is a third, and the
// line lies at half as many voxels (12 coils, 10,240: 47 / 14 and 52 / 19).
constexpr int kShared = 8;
__device__ __forceinline__ int slice_lanes(const DataArgs& a, long long nm) {
    return nm <= 2432LL * (a.nc - 5) / (a.pr.P < 3 ? 2 : 1) ? kShared : 1;
}

// Evaluator codes of the kernels below (with_evaluator): kPadded + NR is eval_padded.
constexpr int kPadded = 100;

// The three-echo path in registers, the padded one, or the general one.
template <typename T, int NC, bool COST, bool CURV>
__device__ __forceinline__ void eval_any(const DataArgs& a, long long j, T w, T& cost, T& grad, T& curv) {
    if constexpr (NC < 0) {
        eval_slice<1, COST>(a, j, 0, w, cost, grad, curv);
    } else if constexpr (NC > kPadded) {
        eval_padded<NC - kPadded, COST, CURV>(a, j, w, cost, grad, curv);
    } else if constexpr (sizeof(T) == 4 && NC > 1) {
        eval_fixed<T, NC, 3, COST, CURV>(a, j, w, cost, grad, curv);
    } else {
        if (NC != 0 && a.L == 3) eval_fixed<T, (NC == 0 ? 1 : NC), 3, COST, CURV>(a, j, w, cost, grad, curv);
        else eval_voxel<T, NC, COST, CURV>(a, j, w, cost, grad, curv);
    }
}

// ------------------------------------------------------------------ gradient pass

// w_out = w_in + alpha z (the previous iteration's update, Algorithm box), then at w_out:
// g = grad Psi (Eq. 8), d (Eq. 10), and Psi (Eq. 5) reduced to scal[S_COST] / cost_hist.
// Runs over the compact list of mask voxels; entries outside the mask are never written
// (the host zeroes them once).
template <typename T, int NC>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 4 && NC == 1 ? 4 : 2) k_grad(DataArgs a) {
    __shared__ double sbuf[32];
    const int nx = a.geo.nx;
    const long long nxy = (long long)nx * a.geo.ny;
    const T* w_in = (const T*)a.w_in;
    const T* z = (const T*)a.z;
    T* w_out = (T*)a.w_out;
    T* g = (T*)a.g;
    T* d = (T*)a.d;
    const T alpha = z ? (T)a.scal[S_ALPHA] : T(0);
    const T beta = (T)a.beta;
    auto upd = [&](long long k) -> T { return z ? w_in[k] + alpha * z[k] : w_in[k]; };
    const long long nm = a.istate[I_NMASK];
    // the thread's cost and penalty sums in T with Kahan compensation, converted to double
    // once (per-voxel FP64 additions would queue on GB300's narrow FP64 pipe)
    T cs = 0, cc = 0, rs = 0, rc = 0;
    auto pass = [&](auto lanes) {
        constexpr int SP = decltype(lanes)::value, VW = 32 / SP;  // lanes per voxel, voxels per warp
        const int lane = threadIdx.x & 31, sl = lane / VW;
        const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
        const long long first = SP == 1 ? tid : tid / 32 * VW, stride = (long long)gridDim.x * blockDim.x / SP;
        for (long long kb = first; kb < nm; kb += stride) {  // SP > 1: the same trips for a whole warp
            const long long k = SP == 1 ? kb : min(kb + lane % VW, nm - 1);
            const bool mine = SP == 1 || (sl == 0 && kb + lane % VW < nm);
            constexpr bool kRegs = sizeof(T) == 4 && NC > 1 && NC < kPadded;  // three echoes, dispatched by coil count
            VoxelData<T, kRegs ? NC : 1, 3, kRegs> data;
            if constexpr (kRegs) data.load(a, k);  // in flight under the stencil's gathers
            const long long j = a.vlist[k];
            const T wj = upd(j);
            T lap = 0, reg = 0;
            if (mine) {
                const uint8_t b = a.nb[j];
                w_out[j] = wj;
                if (b & NB_XM) lap += wj - upd(j - 1);
                if (b & NB_YM) lap += wj - upd(j - nx);
                if (b & NB_ZM) lap += wj - upd(j - nxy);
                if (b & NB_XP) { const T e = wj - upd(j + 1); lap += e; reg += e * e; }
                if (b & NB_YP) { const T e = wj - upd(j + nx); lap += e; reg += e * e; }
                if (b & NB_ZP) { const T e = wj - upd(j + nxy); lap += e; reg += e * e; }
            }
            T cst, gr, cu;
            if constexpr (SP > 1) {
                eval_slice<SP, true>(a, k, sl, wj, cst, gr, cu);
                cst = slice_sum<SP>(cst);
                gr = slice_sum<SP>(gr);
                cu = slice_sum<SP>(cu);
                if (!mine) continue;
            } else if constexpr (kRegs) {
                data.template eval<true>(a, wj, cst, gr, cu);
            } else {
                eval_any<T, NC, true, true>(a, k, wj, cst, gr, cu);
            }
            if (g) g[j] = gr + beta * lap;
            if (d) d[j] = cu;
            {
                const T y1 = cst - cc, t1 = cs + y1;
                cc = (t1 - cs) - y1;
                cs = t1;
                const T y2 = reg - rc, t2 = rs + y2;
                rc = (t2 - rs) - y2;
                rs = t2;
            }
        }
    };
    if (NC < 0 && slice_lanes(a, nm) > 1) pass(std::integral_constant<int, NC < 0 ? kShared : 1>());
    else pass(std::integral_constant<int, 1>());
    double v[1] = {((double)cs - (double)cc) + 0.5 * a.beta * ((double)rs - (double)rc)}, out[1];
    if (last_block_reduce<1>(v, a.partials, (unsigned*)(a.istate + I_DONE0), out, sbuf)) {
        if (threadIdx.x == 0) {
            const double total = a.scal[S_K] + out[0];
            a.scal[S_COST] = total;
            if (a.cost_hist) a.cost_hist[a.istate[I_ITER]] = total;
            if (!isfinite(total)) set_err(a.istate, FM_ERR_NONFINITE);
        }
    }
}

// ------------------------------------------------------------------ line search

// The search direction and the monotonic line search (Algorithm box, Sec. III-C, Eq. 16) as
// one persistent cooperative kernel.
//
// Direction: mu (Polak-Ribiere with the preconditioned gradients; 0 at the first iteration),
// z = -p + mu z, and the sums the line search needs: ||C z||^2, (C z)'(C w), z'g and
// sum z^2 d (each thread sums its voxels in the voxel type, blocks and the grid in FP64, in a
// fixed order, so every block computes the same totals after one grid barrier).  The first
// step alpha_1 = -z'g / (sum z^2 d + beta ||C z||^2) reuses the gradient pass's g and d.
//
// Steps k = 1 .. nls-1: each re-evaluates the data term at w + alpha_k z, reduces
// sum z_j dPhi_j and sum z_j^2 d_j the same way, and updates alpha without leaving the device.
// The direction phase leaves each voxel's (z, w) in compact order (a.zw), so that a step's loads
// all follow from the loop index: with z and w behind the voxel list, and the data term's loads
// behind a test of z, a voxel cost three dependent memory round trips before its arithmetic
// (256 x 256 x 128, eight coils: 722 -> 681 us).  Every thread visits the same voxels in both
// phases (one grid-stride mapping), so it reads back only what it wrote itself -- but for the
// lane-shared form, where the grid barrier between the phases orders the two.
//
// The grid is sized for the whole voxel grid, but a small mask does not need all of it: only
// the first nb blocks take part -- one mask voxel per thread at most (fewer threads with
// several voxels each measured slower: each voxel is a chain of dependent gathers) -- and the
// rest leave before the first grid barrier, which then counts the nb participants only.
// Resident blocks per SM of the line search: compiled for, and the most that its grid takes
// (ls_max_blocks_per_sm), as each thread's voxels and the order of every sum follow from the grid and
// should not from the compiler's register count.  128 registers for eight coils in registers and more than
// eight coils (whose polynomial constants otherwise do not stay in registers), 64 to 80 for the others.
template <typename T, int NC> constexpr int ls_blocks() {
    constexpr int n = sizeof(T) == 8 ? (NC == 0 ? 3 : 2) : NC == 8 || NC < 0 || NC > kPadded + 4 ? 2 : NC > kPadded ? 3 : 4;
    static_assert(n <= kLsMaxBlocks, "a context's partials buffer holds kLsMaxBlocks blocks per SM");
    return n;
}

template <typename T, int NC>
__global__ void __launch_bounds__(kThreads, ls_blocks<T, NC>()) k_ls(DataArgs a) {
    static_assert(kThreads == 256, "block_sum_256");
    __shared__ double s_val[4 * kTree];
    __shared__ double s_tot[4];
    __shared__ T s_aT, s_muT;
    __shared__ double s_mu, s_alpha, s_cz2, s_czw;  // thread 0's, kept out of the other threads' registers
    __shared__ int s_bar;                           // number of the next grid barrier
    const T* w = (const T*)a.w_out;
    using T2 = typename V2<T>::t;
    T2* zw = (T2*)a.zw;
    const int it = a.istate[I_ITER];
    const long long nm = a.istate[I_NMASK];
    const int sp = NC < 0 ? slice_lanes(a, nm) : 1;  // lanes per voxel
    const int nb = (int)max(1LL, min((long long)gridDim.x, (nm * sp + kThreads - 1) / kThreads));
    if ((int)blockIdx.x >= nb) return;
    const int nx = a.geo.nx;
    const long long nxy = (long long)nx * a.geo.ny;
    const int lane0 = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // mu, and each step's alpha below, come from one thread: a double division by all eight warps
    // would hold the FP64 pipe for more than a microsecond
    if (threadIdx.x == 0) {
        double mu = 0.0;
        s_bar = a.istate[I_LS_PH];
        if (it > 0) {
            const double den = a.scal[S_GP_PREV];
            mu = den != 0.0 ? (a.scal[S_GP] - a.scal[S_GPREVP]) / den : 0.0;
        }
        s_mu = mu;
        s_muT = (T)mu;
    }
    __syncthreads();
    {
        const T muT = s_muT;
        const T* p = (const T*)a.p;
        const T* zo = (const T*)a.z_old;
        T* zn = (T*)a.z_new;
        const T* g = (const T*)a.g;
        const T* d = (const T*)a.d;
        auto zval = [&](long long k) -> T { return -p[k] + muT * zo[k]; };
        T t_cz2 = 0, t_czw = 0, t_zg = 0, t_zzd = 0;
        // one voxel's direction entry and its terms of the four sums (the +x, +y, +z edges)
        auto dir_voxel = [&](long long k, long long j, uint8_t b, T pj, T zoj, T wj, T gj, T dj) {
            const T zj = -pj + muT * zoj;
            zn[j] = zj;
            zw[k] = T2{zj, wj};
            if (b & NB_XP) { const T e = zj - zval(j + 1), f = wj - w[j + 1]; t_cz2 += e * e; t_czw += e * f; }
            if (b & NB_YP) { const T e = zj - zval(j + nx), f = wj - w[j + nx]; t_cz2 += e * e; t_czw += e * f; }
            if (b & NB_ZP) { const T e = zj - zval(j + nxy), f = wj - w[j + nxy]; t_cz2 += e * e; t_czw += e * f; }
            t_zg += zj * gj;
            t_zzd += zj * zj * dj;
        };
        // four voxels per pass with their own loads issued first (the gathers of a voxel
        // depend on its list entry), then the rest one by one, in the same voxel order
        constexpr int U = 4;
        const long long stride = (long long)nb * blockDim.x;
        long long k0 = blockIdx.x * (long long)blockDim.x + threadIdx.x;
        for (; k0 + (U - 1) * stride < nm; k0 += U * stride) {
            long long jj[U];
            uint8_t bb[U];
            T pp[U], zz[U], ww[U], gg[U], dd[U];
#pragma unroll
            for (int u = 0; u < U; ++u) jj[u] = a.vlist[k0 + u * stride];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                bb[u] = a.nb[jj[u]];
                pp[u] = p[jj[u]];
                zz[u] = zo[jj[u]];
                ww[u] = w[jj[u]];
                gg[u] = g[jj[u]];
                dd[u] = d[jj[u]];
            }
#pragma unroll
            for (int u = 0; u < U; ++u) dir_voxel(k0 + u * stride, jj[u], bb[u], pp[u], zz[u], ww[u], gg[u], dd[u]);
        }
        for (long long k = k0; k < nm; k += stride) {
            const long long j = a.vlist[k];
            dir_voxel(k, j, a.nb[j], p[j], zo[j], w[j], g[j], d[j]);
        }
        const double v[4] = {(double)t_cz2, (double)t_czw, (double)t_zg, (double)t_zzd};
        const double bs = block_sum_256<4>(v, s_val);
        if (wid < 4 && lane0 == 0) a.partials[(size_t)wid * nb + blockIdx.x] = bs;
        if (!ls_barrier(a.istate, a.spin_limit, nb, &s_bar)) return;
        if (wid < 4) {
            const double t = sum_partials_256(a.partials + (size_t)wid * nb, nb);
            if (lane0 == 0) s_tot[wid] = t;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double mu = s_mu, cz2 = s_tot[0], czw = s_tot[1];
        const double den = s_tot[3] + a.beta * cz2;
        const double alpha = den != 0.0 ? -s_tot[2] / den : 0.0;
        s_cz2 = cz2;
        s_czw = czw;
        s_alpha = alpha;
        s_aT = (T)alpha;
        if (blockIdx.x == 0) {
            a.scal[S_CZ2] = cz2;
            a.scal[S_CZW] = czw;
            a.scal[S_ZG] = s_tot[2];
            a.scal[S_ZZD] = s_tot[3];
            a.scal[S_MU] = mu;
            a.scal[S_GP_PREV] = a.scal[S_GP];  // every block read the old value before the barrier
            if (a.mu_hist) a.mu_hist[it] = mu;
            if (!isfinite(alpha) || !isfinite(mu) || !isfinite(den)) set_err(a.istate, FM_ERR_NONFINITE);
        }
    }
    __shared__ bool s_stop;
    if (threadIdx.x == 0) s_stop = false;
    __syncthreads();
    for (int step = 1; step < a.nls; ++step) {
        const T aT = s_aT;
        // each thread sums its few voxels in the voxel type, then the block and the grid in FP64
        T t1 = 0, t2 = 0;
        if constexpr (NC == 1) {
            // one coil, or the combined curvature: little arithmetic, so four voxels per pass with
            // their loads issued first, then the rest one by one, in the same voxel order
            constexpr int U = 4;
            const long long stride = (long long)nb * blockDim.x;
            long long k0 = blockIdx.x * (long long)blockDim.x + threadIdx.x;
            for (; k0 + (U - 1) * stride < nm; k0 += U * stride) {
                T2 q[U];
#pragma unroll
                for (int u = 0; u < U; ++u) q[u] = zw[k0 + u * stride];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    T cst, gr, cu;
                    eval_any<T, NC, false, true>(a, k0 + u * stride, q[u].y + aT * q[u].x, cst, gr, cu);
                    t1 += q[u].x * gr;
                    t2 += q[u].x * q[u].x * cu;
                }
            }
            for (long long k = k0; k < nm; k += stride) {
                const T2 q = zw[k];
                T cst, gr, cu;
                eval_any<T, NC, false, true>(a, k, q.y + aT * q.x, cst, gr, cu);
                t1 += q.x * gr;
                t2 += q.x * q.x * cu;
            }
        } else {
            bool shared = false;
            if constexpr (NC < 0) {
                if (sp > 1) {
                    // each slice adds its own share: the sums run over all lanes anyway
                    constexpr int SP = kShared, VW = 32 / SP;  // voxels per warp
                    const int lane = threadIdx.x & 31;
                    const long long warp = (blockIdx.x * (long long)blockDim.x + threadIdx.x) / 32;
                    for (long long k = warp * VW + lane % VW; k < nm; k += (long long)nb * blockDim.x / SP) {
                        const T2 q = __ldcg(zw + k);  // written by another thread before the grid barrier
                        T cst, gr, cu;
                        eval_slice<SP, false>(a, k, lane / VW, q.y + aT * q.x, cst, gr, cu);
                        t1 += q.x * gr;
                        t2 += q.x * q.x * cu;
                    }
                    shared = true;
                }
            }
            // a voxel with z = 0 adds exactly 0
            for (long long k = shared ? nm : blockIdx.x * (long long)blockDim.x + threadIdx.x; k < nm;
                 k += (long long)nb * blockDim.x) {
                const T2 q = zw[k];
                T cst, gr, cu;
                eval_any<T, NC, false, true>(a, k, q.y + aT * q.x, cst, gr, cu);
                t1 += q.x * gr;
                t2 += q.x * q.x * cu;
            }
        }
        const double v[2] = {(double)t1, (double)t2};
        const double bs = block_sum_256<2>(v, s_val);
        double* part = a.partials + 4 * (size_t)nb + (size_t)(step & 1) * 2 * nb;
        if (wid < 2 && lane0 == 0) part[(size_t)wid * nb + blockIdx.x] = bs;
        if (!ls_barrier(a.istate, a.spin_limit, nb, &s_bar)) return;
        if (wid < 2) {
            const double t = sum_partials_256(part + (size_t)wid * nb, nb);
            if (lane0 == 0) s_tot[wid] = t;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double alpha = s_alpha;
            const double fp = s_tot[0] + a.beta * (s_czw + alpha * s_cz2);
            const double den = s_tot[1] + a.beta * s_cz2;
            alpha = den == 0.0 ? 0.0 : alpha - fp / den;
            s_alpha = alpha;
            s_aT = (T)alpha;
            s_stop = den == 0.0;
        }
        __syncthreads();
        if (s_stop) break;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const double alpha = s_alpha;
        a.scal[S_ALPHA] = alpha;
        if (a.alpha_hist) a.alpha_hist[it] = alpha;
        if (!isfinite(alpha)) set_err(a.istate, FM_ERR_NONFINITE);
        a.istate[I_ITER] = it + 1;
        a.istate[I_LS_PH] = s_bar;
    }
}

// ------------------------------------------------------------------ diagonal / no preconditioner

// p = g / H_jj (mode 1, the NCG-MLS-D comparison) or p = g (mode 2), with g'p and g_prev'p.
template <typename T>
__global__ void __launch_bounds__(kThreads) k_pdiag(DataArgs a, int mode) {
    __shared__ double sbuf[2 * 32];
    const T* g = (const T*)a.g;
    const T* gp = (const T*)a.g_prev;
    const T* d = (const T*)a.d;
    T* p = (T*)a.z_new;  // output slot
    double s_gp = 0.0, s_gpp = 0.0;
    const long long nm = a.istate[I_NMASK];
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < nm;
         k += (long long)gridDim.x * blockDim.x) {
        const long long j = a.vlist[k];
        const uint8_t b = a.nb[j];
        T pj = g[j];
        if (mode == 1) {
            const int cnt = __popc((unsigned)(b >> 1) & 0x3fu);
            const T h = d[j] + (T)a.beta * (T)cnt;
            if (!(h > T(0))) set_err(a.istate, FM_ERR_NOT_PD);
            pj = h > T(0) ? pj / h : T(0);
        }
        p[j] = pj;
        s_gp += (double)(g[j] * pj);
        s_gpp += (double)(gp[j] * pj);
    }
    double v[2] = {s_gp, s_gpp}, out[2];
    if (last_block_reduce<2>(v, a.partials, (unsigned*)(a.istate + I_DONE0), out, sbuf)) {
        if (threadIdx.x == 0) {
            a.scal[S_GP] = out[0];
            a.scal[S_GPREVP] = out[1];
        }
    }
}

// ------------------------------------------------------------------ launchers

// Calls f(integral constant NC) with the evaluator of a context: 1 coil-combined curvature (or one
// coil); 2, 4, 8 that many coils and three echoes in registers; kPadded + NR (FP32) other literal
// curvatures of up to NR coils; -8 (FP32) more than eight coils, eight lanes per voxel or one; 0 a runtime
// coil count with one thread per voxel (FP64, and the water-fat model).
template <typename T, typename F>
static auto with_evaluator(const DataArgs& a, F f) {
    if (!a.literal) return f(std::integral_constant<int, 1>());
    if (a.wf) return f(std::integral_constant<int, 0>());
    if (sizeof(T) == 8 || a.L == 3) {
        switch (a.nc) {
            case 2: return f(std::integral_constant<int, 2>());
            case 4: return f(std::integral_constant<int, 4>());
            case 8: return f(std::integral_constant<int, 8>());
            default: break;
        }
    }
    if constexpr (sizeof(T) == 4) {
        if (a.nc <= 2) return f(std::integral_constant<int, kPadded + 2>());
        if (a.nc <= 4) return f(std::integral_constant<int, kPadded + 4>());
        if (a.nc <= 6) return f(std::integral_constant<int, kPadded + 6>());
        if (a.nc <= 8) return f(std::integral_constant<int, kPadded + 8>());
        return f(std::integral_constant<int, -8>());
    }
    return f(std::integral_constant<int, 0>());
}

int data_lanes(const DataArgs& a) {
    return with_evaluator<float>(a, [](auto nc) { return decltype(nc)::value < 0 ? -decltype(nc)::value : 1; });
}

template <typename T>
cudaError_t launch_grad(const DataArgs& a, int grid, cudaStream_t s) {
    return with_evaluator<T>(a, [&](auto nc) {
        k_grad<T, decltype(nc)::value><<<grid, kThreads, 0, s>>>(a);
        return cudaGetLastError();
    });
}

template <typename T>
cudaError_t launch_ls(const DataArgs& a, int grid, cudaStream_t s) {
    return with_evaluator<T>(a, [&](auto nc) {
        DataArgs copy = a;
        void* args[] = {&copy};
        return cudaLaunchCooperativeKernel((const void*)k_ls<T, decltype(nc)::value>, dim3(grid), dim3(kThreads), args, 0, s);
    });
}

template <typename T>
int ls_max_blocks_per_sm(const DataArgs& a) {
    return with_evaluator<T>(a, [&](auto nc) {
        int n = 0;
        const cudaError_t e =
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_ls<T, decltype(nc)::value>, kThreads, 0);
        return e == cudaSuccess ? std::min(n, ls_blocks<T, decltype(nc)::value>()) : 0;
    });
}

template <typename T>
cudaError_t launch_pdiag(const DataArgs& a, int mode, int grid, cudaStream_t s) {
    k_pdiag<T><<<grid, kThreads, 0, s>>>(a, mode);
    return cudaGetLastError();
}

#define FM_INST(T)                                                                  \
    template cudaError_t launch_grad<T>(const DataArgs&, int, cudaStream_t);        \
    template cudaError_t launch_ls<T>(const DataArgs&, int, cudaStream_t);          \
    template cudaError_t launch_pdiag<T>(const DataArgs&, int, int, cudaStream_t);  \
    template int ls_max_blocks_per_sm<T>(const DataArgs&);
FM_INST(float)
FM_INST(double)

}  // namespace fm
