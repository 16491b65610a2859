// Offline encoder steps on the GPU (the step before the hot path): groupwise code assignment,
// closed-form scale, the two reconstruction losses, and the deterministic candidate search, under
// the continuous objective of Section 4.1 or the dual-path objective L_C + L_A8 of Section 4.3.
//
// Decisions (which code, which candidate) are taken in fp64, the precision the method is stated in;
// the carrier grid uses the pinned fp32 sequence of Eq. carrier.  This file is compiled without
// floating-point contraction so that a product followed by a sum rounds twice, as written.
//
// One lane owns one candidate of one group in the search kernel; the assignment / scale / loss kernels use one
// block per group.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "../../include/cubicquant.h"
#include "cq_internal.h"

namespace cq {
namespace {

constexpr int MAXL = 128;      // most non-negative levels (W8)

__device__ __forceinline__ int top_code(int B) { return (1 << (B - 1)) - 1; }   // M of Eq. codes
__device__ __forceinline__ double half_bits_to_double(uint16_t h) { return (double)__half2float(__ushort_as_half(h)); }
__device__ __forceinline__ uint16_t double_to_half_bits(double v) { return __half_as_ushort(__double2half(v)); }

// q(t) = t [a + t (b + c t)], c = 1 - a - b (Eq. cubic)
__device__ __forceinline__ double level_curve(double t, double a, double b) {
    const double c = 1.0 - a - b;
    return t * (a + t * (b + t * c));
}

// m(a, b) = min over [0, 1] of q'(t) (Eq. shape-domain): the end points, and the vertex of the
// quadratic when it lies inside the interval and opens upwards
__host__ __device__ inline double shape_margin(double a, double b) {
    const double c = 1.0 - a - b;
    double m = fmin(a, 3.0 - 2.0 * a - b);
    if (c > 0.0 && b < 0.0 && b > -3.0 * c) m = fmin(m, a - b * b / (3.0 * c));
    return m;
}

// carrier-grid levels round(127 q) / 127 of a shape given in fp32 (Eq. carrier-grid), the rounding by
// the pinned fp32 sequence t = i / M, c = (1 - a) - b, q = t fma(t, fma(t, c, b), a), RNE(127 q)
__device__ __noinline__ void carrier_grid(int B, float a, float b, double *zt) {
    const int M = top_code(B);
    if (B == 2) { zt[0] = 0.0; zt[1] = 1.0; return; }
    const float c = __fsub_rn(__fsub_rn(1.0f, a), b);
    for (int i = 0; i <= M; ++i) {
        const float t = __fdiv_rn((float)i, (float)M);
        const float q = __fmul_rn(t, fmaf(t, fmaf(t, c, b), a));
        int r = __float2int_rn(__fmul_rn(127.0f, q));
        r = min(max(r, 0), 127);
        zt[i] = (double)r / 127.0;
    }
}

// nearest level among increasing y_0 .. y_M, ties to the lower index, saturating at M
__device__ __forceinline__ int nearest_level(double u, const double *y, int M) {
    int lo = 0, hi = M;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (u <= 0.5 * (y[mid] + y[mid + 1])) hi = mid; else lo = mid + 1;
    }
    return lo;
}

// minimiser of (u - s z_i)^2 + (u - s zt_i)^2 (Eq. carrier-aware-assignment), first minimum wins
__device__ __forceinline__ int joint_level(double u, double s, const double *z, const double *zt, int M) {
    int best = 0;
    double bc = INFINITY;
    for (int i = 0; i <= M; ++i) {
        const double d1 = u - s * z[i], d2 = u - s * zt[i];
        const double cst = d1 * d1 + d2 * d2;
        if (cst < bc) { bc = cst; best = i; }
    }
    return best;
}

// ------------------------------------------------------------------ per-group kernels (one block per group)
__global__ void __launch_bounds__(128) assign_kernel(const float *__restrict__ W, int B, int G, int64_t K, int64_t ng,
                                                     const float *__restrict__ scale, const uint16_t *__restrict__ a,
                                                     const uint16_t *__restrict__ b, int joint, int8_t *__restrict__ k) {
    __shared__ double z[MAXL], zt[MAXL], y[MAXL];
    const int64_t gi = blockIdx.x, n = gi / ng, g = gi % ng;
    const float *w = W + n * K + g * G;
    int8_t *ko = k + n * K + g * G;
    if (B == 1) {
        for (int j = threadIdx.x; j < G; j += blockDim.x) ko[j] = (int8_t)(w[j] >= 0.0f ? 1 : -1);
        return;
    }
    const int M = top_code(B);
    const double s = (double)scale[gi], av = half_bits_to_double(a[gi]), bv = half_bits_to_double(b[gi]);
    for (int i = threadIdx.x; i <= M; i += blockDim.x) {
        z[i] = level_curve((double)i / (double)M, av, bv);
        y[i] = s * z[i];
    }
    if (joint && threadIdx.x == 0) carrier_grid(B, (float)av, (float)bv, zt);
    __syncthreads();
    for (int j = threadIdx.x; j < G; j += blockDim.x) {
        const double u = fabs((double)w[j]);
        const int i = joint ? joint_level(u, s, z, zt, M) : nearest_level(u, y, M);
        ko[j] = (int8_t)(w[j] < 0.0f ? -i : i);
    }
}

// sums of a block in a fixed order: each thread adds its strided elements, then thread 0 adds the
// per-thread sums in thread order
__device__ double block_sum(double v, double *sh) {
    sh[threadIdx.x] = v;
    __syncthreads();
    double tot = 0.0;
    if (threadIdx.x == 0) for (int i = 0; i < (int)blockDim.x; ++i) tot += sh[i];
    __syncthreads();
    return tot;   // valid in thread 0
}

// scale[g] = sum u (z + zt) / sum (z^2 + zt^2) (Eq. carrier-aware-scale), or the continuous analogue
__global__ void __launch_bounds__(128) scale_kernel(const float *__restrict__ W, const int8_t *__restrict__ k, int B, int G,
                                                    int64_t K, int64_t ng, const uint16_t *__restrict__ a,
                                                    const uint16_t *__restrict__ b, int joint, float *__restrict__ scale) {
    __shared__ double z[MAXL], zt[MAXL], sh[128];
    const int64_t gi = blockIdx.x, n = gi / ng, g = gi % ng;
    const float *w = W + n * K + g * G;
    const int8_t *kk = k + n * K + g * G;
    const int M = B == 1 ? 1 : top_code(B);
    if (B > 1) {
        const double av = half_bits_to_double(a[gi]), bv = half_bits_to_double(b[gi]);
        for (int i = threadIdx.x; i <= M; i += blockDim.x) z[i] = level_curve((double)i / (double)M, av, bv);
        if (threadIdx.x == 0) {
            if (joint) carrier_grid(B, (float)av, (float)bv, zt);
            else for (int i = 0; i <= M; ++i) zt[i] = 0.0;
        }
    }
    __syncthreads();
    double num = 0.0, den = 0.0;
    for (int j = threadIdx.x; j < G; j += blockDim.x) {
        const double u = fabs((double)w[j]);
        if (B == 1) { num += u; den += 1.0; continue; }
        const int c = kk[j];
        const int i = (c == -(1 << (B - 1))) ? 0 : abs(c);
        if (joint) { num += u * (z[i] + zt[i]); den += z[i] * z[i] + zt[i] * zt[i]; }
        else { num += u * z[i]; den += z[i] * z[i]; }
    }
    const double tn = block_sum(num, sh), td = block_sum(den, sh);
    if (threadIdx.x == 0) scale[gi] = td > 0.0 ? (float)(tn / td) : 0.0f;
}

// L_C = sum (w - s q)^2 and L_A8 = sum (w - (s / 127) r)^2 per group (Eq. continuous-and-carrier-loss)
__global__ void __launch_bounds__(128) losses_kernel(const float *__restrict__ W, const int8_t *__restrict__ k, int B, int G,
                                                     int64_t K, int64_t ng, const float *__restrict__ scale,
                                                     const uint16_t *__restrict__ a, const uint16_t *__restrict__ b,
                                                     double *__restrict__ LC, double *__restrict__ LA8) {
    __shared__ double z[MAXL], zt[MAXL], sh[128];
    const int64_t gi = blockIdx.x, n = gi / ng, g = gi % ng;
    const float *w = W + n * K + g * G;
    const int8_t *kk = k + n * K + g * G;
    const double s = (double)scale[gi];
    const int M = B == 1 ? 1 : top_code(B);
    if (B > 1) {
        const double av = half_bits_to_double(a[gi]), bv = half_bits_to_double(b[gi]);
        for (int i = threadIdx.x; i <= M; i += blockDim.x) z[i] = level_curve((double)i / (double)M, av, bv);
        if (threadIdx.x == 0) carrier_grid(B, (float)av, (float)bv, zt);
    }
    __syncthreads();
    double lc = 0.0, la = 0.0;
    for (int j = threadIdx.x; j < G; j += blockDim.x) {
        const int c = kk[j];
        const double wv = (double)w[j];
        if (B == 1) { const double d = wv - (c > 0 ? 1.0 : -1.0) * s; lc += d * d; la += d * d; continue; }
        const int i = (c == -(1 << (B - 1))) ? 0 : abs(c);
        const double sg = c < 0 ? -1.0 : 1.0;
        const double d1 = wv - sg * s * z[i], d2 = wv - sg * s * zt[i];
        lc += d1 * d1; la += d2 * d2;
    }
    const double tc = block_sum(lc, sh), ta = block_sum(la, sh);
    if (threadIdx.x == 0) { LC[gi] = tc; LA8[gi] = ta; }
}

// ------------------------------------------------------------------ the candidate search
// The candidates of a group (a start shape, a start scale, some rounds) do not depend on one another until the
// best is picked, so one LANE runs one candidate of one group and a block holds all candidates of a few groups:
// forty-five of them at effort "fast", twice that under the joint objective.  Bound: the fp64 pipe and the issue slots
// around it.  2048 x 4096, W4 G128, joint, with packing and layout: 222 ms with one thread per group (its levels and
// indices in local memory, 14 warps per SM, M + 1 costs per weight), 16.7 ms so.  The sums over a group must be
// taken in the order of its weights (they decide codes), so a lane walks its group alone; the weights sit in
// shared memory and are the same address for the lanes of a group.  What a lane keeps per level (z, the carrier grid,
// the guard) sits in its own column of shared memory, [level][thread], free of bank conflicts for any index.
//
// Code assignment is a comparison against M thresholds, no search over the levels:
//   continuous   u <= (y_i + y_(i+1)) / 2 for an fp32 u holds exactly when u <= that midpoint rounded down to fp32;
//   joint        the cost of level i, (u - s z_i)^2 + (u - s zt_i)^2, is 2 u^2 plus a line in u whose slope falls
//                with i, so the best level changes at u = s beta_i, beta_i = (dz mz + dzt mzt) / (dz + dzt) with d the
//                step and m the midpoint between neighbours.  Thresholds are formed in fp32; a weight within
//                GUARD s = 4e-6 s of one (beta s <= s carries a few rounding errors of 2^-24 s = 6e-8 s), and any lane
//                whose levels or scale do not meet the conditions of joint_thresholds, takes the definition
//                (joint_level), so the codes are those of the definition everywhere.
struct SearchPlan {      // what the host fixes for a launch
    int G, groups_per_block, n_int, n_shape, clips, iters, refine, dual;
    int64_t groups;
    double shapes[144][2];
    double clip[6];
};
constexpr int INT_CLIPS = 15;
constexpr float GUARD = 4e-6f;
struct __align__(16) Weight { double u; float f; int pad; };   // |w| as fp64 and as the fp32 it came from

template <int B>
struct SearchShape {
    static constexpr int M = (1 << (B - 1)) - 1, L = M + 1, T = 128;
    // Up to sixteen levels: levels and carrier grid in tables, thresholds in registers, bisected by selects.  More: a lane's
    // column would be kilobytes, so it holds the thresholds (bisected where they lie) and the carriers as bytes, and a level is
    // computed again when it is read.
    static constexpr bool TAB = B <= 5;
    static constexpr int COL = TAB ? L * (8 + 8 + 4) : L * (4 + 1);      // bytes of a lane's column
    static constexpr int FINAL = (T / 32) * L * 16;                      // level tables of the last step, one set per warp
};
// a lane's view of shared memory
template <int B>
struct Columns {
    using S = SearchShape<B>;
    double *z_, *zt_;        // [L][T], TAB: levels and carrier-grid levels
    float *above;            // [L][T], TAB, joint: entry i = lower end of level i's safe range
    float *thr;              // [M][T], otherwise: thresholds
    uint8_t *carrier;        // [L][T], otherwise
    const double *td;        // i / M
    const double *phi;       // [3][L]: t^3, t - t^3, t^2 - t^3
    const float *tf;         // i / M in fp32
    const double *r127;      // r / 127
    double a, b;             // the shape whose levels are in place
    __device__ __forceinline__ double z(int i) const { if constexpr (S::TAB) return z_[i * S::T]; else return level_curve(td[i], a, b); }
    __device__ __forceinline__ double zt(int i) const { if constexpr (S::TAB) return zt_[i * S::T]; else return r127[carrier[i * S::T]]; }
};
// and what it keeps in registers
template <int B>
struct Lane : Columns<B> {
    float reg[SearchShape<B>::TAB ? SearchShape<B>::M : 1];
    float guard2;            // joint: width of the guard around a threshold
    bool exact_only;         // joint: every weight by the definition
    __device__ __forceinline__ explicit Lane(const Columns<B> &c) : Columns<B>(c), guard2(0.0f), exact_only(false) {}
};

template <int B, bool JOINT>
__device__ __forceinline__ void set_levels(Lane<B> &ln, double a, double b) {
    using S = SearchShape<B>;
    ln.a = a; ln.b = b;
    if constexpr (S::TAB) {
#pragma unroll 1
        for (int i = 0; i < S::L; ++i) ln.z_[i * S::T] = level_curve(ln.td[i], a, b);
    }
    if constexpr (JOINT) {   // carrier_grid, its two divisions read from tables of the same quotients
        const float af = (float)a, bf = (float)b, c = __fsub_rn(__fsub_rn(1.0f, af), bf);
#pragma unroll 1
        for (int i = 0; i < S::L; ++i) {
            const float t = ln.tf[i];
            const float q = __fmul_rn(t, fmaf(t, fmaf(t, c, bf), af));
            const int r = min(max(__float2int_rn(__fmul_rn(127.0f, q)), 0), 127);
            if constexpr (S::TAB) ln.zt_[i * S::T] = ln.r127[r]; else ln.carrier[i * S::T] = (uint8_t)r;
        }
    }
}

// Thresholds of the continuous assignment under scale s: exact (see above).
template <int B>
__device__ __forceinline__ void continuous_thresholds(Lane<B> &ln, double s) {
    using S = SearchShape<B>;
    double y0 = s * ln.z(0);
    auto at = [&](int i) {
        const double y1 = s * ln.z(i + 1);
        const float t = __double2float_rd(0.5 * (y0 + y1));
        y0 = y1;
        return t;
    };
    if constexpr (S::TAB) {
#pragma unroll
        for (int i = 0; i < S::M; ++i) ln.reg[i] = at(i);
    } else {
#pragma unroll 1
        for (int i = 0; i < S::M; ++i) ln.thr[i * S::T] = at(i);
    }
}
// Thresholds of the joint assignment.  They are used where: s is far from the ends of the fp32 range and the largest
// weight within 10^6 s; every step dz + dzt is at least 1e-5 (then a weight outside the guard prefers one level to
// its neighbour by more than 2 s^2 1e-5 GUARD, against 1e-15 of costs of at most 2 u^2 in rounding); and the thresholds
// rise by more than the guard, so that the preference between neighbours orders all levels.
template <int B>
__device__ __forceinline__ void joint_thresholds(Lane<B> &ln, double s, float umax) {
    using S = SearchShape<B>;
    const float sf = (float)s, guard = GUARD * sf;
    bool ok = sf > 1e-25f && sf < 1e25f && umax < 1e6f * sf;
    double z0 = ln.z(0), t0 = ln.zt(0);
    float last = -1e30f;
    ln.guard2 = 2.0f * guard;
    if constexpr (S::TAB) ln.above[0] = -1.0f;
    auto at = [&](int i) {
        const double z1 = ln.z(i + 1), t1 = ln.zt(i + 1);
        const float dz = (float)(z1 - z0), dt = (float)(t1 - t0), mz = 0.5f * (float)(z1 + z0), mt = 0.5f * (float)(t1 + t0);
        const float d = dz + dt, beta = mz + (mt - mz) * __fdividef(dt, d);
        z0 = z1; t0 = t1;
        ok = ok && dz > 0.0f && dt >= 0.0f && d > 1e-5f && beta > last + 4.0f * GUARD;
        last = beta;
        if constexpr (S::TAB) ln.above[(i + 1) * S::T] = fmaf(beta, sf, guard);
        return fmaf(beta, sf, -guard);
    };
    if constexpr (S::TAB) {
#pragma unroll
        for (int i = 0; i < S::M; ++i) ln.reg[i] = at(i);
    } else {
#pragma unroll 1
        for (int i = 0; i < S::M; ++i) ln.thr[i * S::T] = at(i);
    }
    ln.exact_only = !ok;
}
template <int B, bool JOINT>
__device__ __forceinline__ void set_thresholds(Lane<B> &ln, double s, float umax) {
    if constexpr (JOINT) joint_thresholds(ln, s, umax); else continuous_thresholds(ln, s);
}

template <int B>
__device__ __noinline__ int joint_level_exact(Columns<B> ln, double u, double s) {   // joint_level on a lane's own levels
    int best = 0;
    double bc = INFINITY;
#pragma unroll 1
    for (int i = 0; i <= SearchShape<B>::M; ++i) {
        const double d1 = u - s * ln.z(i), d2 = u - s * ln.zt(i);
        const double cst = d1 * d1 + d2 * d2;
        if (cst < bc) { bc = cst; best = i; }
    }
    return best;
}
// the level of one weight by the thresholds; sure: false if it has to be found by the definition
template <int B, bool JOINT>
__device__ __forceinline__ int threshold_level(const Lane<B> &ln, const Weight &w, bool &sure) {
    using S = SearchShape<B>;
    int i = 0;
    if constexpr (S::TAB) {
        // the bisection of nearest_level, its thresholds picked by selects: M = 2^d - 1 of them take d comparisons and M - d
        // selects, against M comparisons and M additions one by one
        float c[S::M];
#pragma unroll
        for (int k = 0; k < S::M; ++k) c[k] = ln.reg[k];
#pragma unroll
        for (int n = S::M; n > 0; n >>= 1) {
            const int h = n >> 1;
            const bool up = JOINT ? w.f > c[h] : !(w.f <= c[h]);
            i += up ? h + 1 : 0;
#pragma unroll
            for (int k = 0; k < h; ++k) c[k] = up ? c[h + 1 + k] : c[k];
        }
    } else {
        int lo = 0, hi = S::M;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            const float t = ln.thr[mid * S::T];
            if (JOINT ? !(w.f > t) : w.f <= t) hi = mid; else lo = mid + 1;
        }
        i = lo;
    }
    sure = true;
    if constexpr (JOINT) {
        float lower;
        if constexpr (S::TAB) lower = ln.above[i * S::T];
        else lower = i > 0 ? ln.thr[(i - 1) * S::T] + ln.guard2 : -1.0f;
        sure = w.f > lower;
    }
    return i;
}
// f(weight, level) for the weights of a group in their order, STEP at a time: one branch for those that need the definition, and
// their look-ups overlap.  (With the bisection above: 2048 x 4096, G = 128, joint, W4 23.5 -> 16.7 ms with four, 17.4 with two; W5
// 41.3 -> 25 with two; four at W5 spill.)
template <int B, bool JOINT, class F>
__device__ __forceinline__ void for_levels(const Lane<B> &ln, const Weight *w, int G, double s, F &&f) {
    constexpr int STEP = B == 3 || B == 5 ? 2 : 4;   // G is a multiple of 32
#pragma unroll 1
    for (int j = 0; j < G; j += STEP) {
        Weight x[STEP];
        int i[STEP];
        bool sure[STEP], all = !JOINT || !ln.exact_only;
#pragma unroll
        for (int e = 0; e < STEP; ++e) {
            x[e] = w[j + e];
            i[e] = threshold_level<B, JOINT>(ln, x[e], sure[e]);
            all = all && sure[e];
        }
        if (JOINT && !all) {
#pragma unroll
            for (int e = 0; e < STEP; ++e) if (ln.exact_only || !sure[e]) i[e] = joint_level_exact<B>(ln, x[e].u, s);
        }
#pragma unroll
        for (int e = 0; e < STEP; ++e) f(x[e], i[e]);
    }
}
// closed-form scale under the assignment that the thresholds in place give
template <int B, bool JOINT>
__device__ __forceinline__ double assigned_scale(const Lane<B> &ln, const Weight *w, int G, double s) {
    double num = 0.0, den = 0.0;
    for_levels<B, JOINT>(ln, w, G, s, [&](const Weight &x, int i) {
        const double z = ln.z(i);
        if constexpr (JOINT) {
            const double zt = ln.zt(i);
            num += x.u * (z + zt); den += z * z + zt * zt;
        } else {
            num += x.u * z; den += z * z;
        }
    });
    return den > 0.0 ? num / den : s;
}

// Score what would be stored (Section 4.1, end; Section 4.3 for the joint objective): a, b to binary16,
// s to binary32, strictly monotone curve required, assignment repeated under the rounded parameters,
// the scale re-fitted and re-rounded once, assignment repeated, loss of the stored representation.
struct Fit { double loss; float s; uint16_t a16, b16; };   // loss = infinity: not a valid representation
template <int B, bool JOINT>
__device__ __forceinline__ Fit score_serialised(Lane<B> &ln, const Weight *w, int G, float umax, double s, double a, double b) {
    using S = SearchShape<B>;
    Fit f; f.loss = INFINITY; f.s = 0.0f;
    f.a16 = double_to_half_bits(a); f.b16 = double_to_half_bits(b);
    const double ar = half_bits_to_double(f.a16), br = half_bits_to_double(f.b16);
    if (!(s > 0.0) || !isfinite(s)) return f;
    if (!(shape_margin(ar, br) > 0.0)) return f;
    set_levels<B, JOINT>(ln, ar, br);
    bool rising = true;
#pragma unroll 1
    for (int i = 0; i < S::M; ++i) rising = rising && ln.z(i + 1) > ln.z(i);
    if (!rising) return f;
    float s32 = (float)s;
    set_thresholds<B, JOINT>(ln, (double)s32, umax);
    const double s2 = assigned_scale<B, JOINT>(ln, w, G, (double)s32);
    if (s2 > 0.0 && isfinite(s2)) s32 = (float)s2;
    if (!(s32 > 0.0f)) return f;
    const double sd = (double)s32;
    set_thresholds<B, JOINT>(ln, sd, umax);
    double loss = 0.0;
    for_levels<B, JOINT>(ln, w, G, sd, [&](const Weight &x, int i) {
        const double d = x.u - sd * ln.z(i);
        loss += d * d;
        if constexpr (JOINT) { const double d2 = x.u - sd * ln.zt(i); loss += d2 * d2; }
    });
    f.s = s32;
    f.loss = loss < INFINITY ? loss : INFINITY;   // NaN never wins
    return f;
}

// 3 x 3 symmetric normal equations by Gaussian elimination with partial pivoting (row permutation kept in perm)
__device__ __noinline__ bool solve_3x3(double A[3][3], double r[3], double p[3]) {
    int perm[3] = {0, 1, 2};
    for (int c = 0; c < 3; ++c) {
        int piv = c;
        for (int i = c + 1; i < 3; ++i) if (fabs(A[perm[i]][c]) > fabs(A[perm[piv]][c])) piv = i;
        const int t = perm[c]; perm[c] = perm[piv]; perm[piv] = t;
        const double dd = A[perm[c]][c];
        if (fabs(dd) < 1e-300) return false;
        for (int i = c + 1; i < 3; ++i) {
            const double f = A[perm[i]][c] / dd;
            for (int j = c; j < 3; ++j) A[perm[i]][j] -= f * A[perm[c]][j];
            r[perm[i]] -= f * r[perm[c]];
        }
    }
    for (int c = 2; c >= 0; --c) {
        double acc = r[perm[c]];
        for (int j = c + 1; j < 3; ++j) acc -= A[perm[c]][j] * p[j];
        p[c] = acc / A[perm[c]][c];
    }
    return true;
}

// One candidate: from shape (a, b) and scale s0 alternate assignment and fitted scale `iters` times,
// then `refine` rounds in which, with the assignment held, the levels s (t^3 + a (t - t^3) + b (t^2 - t^3))
// (Eq. affine-cubic-level) are fitted by the 3 x 3 normal equations in (s, s a, s b); a step is kept
// only while the curve stays strictly monotone with some margin.  A round that returns the parameters it
// started from would do so for ever: the rounds left are not run.
template <int B, bool JOINT>
__device__ __noinline__ Fit try_candidate(Columns<B> columns, const Weight *w, int G, float umax, double a, double b, double s0, int iters, int refine) {
    using S = SearchShape<B>;
    Lane<B> ln(columns);
    double s = s0;
    set_levels<B, JOINT>(ln, a, b);
#pragma unroll 1
    for (int it = 0; it < iters; ++it) {
        set_thresholds<B, JOINT>(ln, s, umax);
        const double sn = assigned_scale<B, JOINT>(ln, w, G, s);
        if (sn == s) break;
        s = sn;
    }
#pragma unroll 1
    for (int rf = 0; rf < refine; ++rf) {
        if (rf > 0) set_levels<B, JOINT>(ln, a, b);
        set_thresholds<B, JOINT>(ln, s, umax);
        double A00 = 0.0, A01 = 0.0, A02 = 0.0, A11 = 0.0, A12 = 0.0, A22 = 0.0, r0 = 0.0, r1 = 0.0, r2 = 0.0;
        for_levels<B, JOINT>(ln, w, G, s, [&](const Weight &x, int i) {
            const double p0 = ln.phi[i], p1 = ln.phi[S::L + i], p2 = ln.phi[2 * S::L + i];
            r0 += p0 * x.u; r1 += p1 * x.u; r2 += p2 * x.u;
            A00 += p0 * p0; A01 += p0 * p1; A02 += p0 * p2;
            A11 += p1 * p1; A12 += p1 * p2; A22 += p2 * p2;
        });
        double A[3][3] = {{A00, A01, A02}, {A01, A11, A12}, {A02, A12, A22}}, r[3] = {r0, r1, r2}, p[3];
        if (!solve_3x3(A, r, p)) break;
        if (!(p[0] > 0.0) || !isfinite(p[0])) break;
        const double an = p[1] / p[0], bn = p[2] / p[0];
        if (!isfinite(an) || !isfinite(bn) || !(shape_margin(an, bn) > 1e-3)) break;
        if (fabs(an) > 8.0 || fabs(bn) > 8.0) break;
        const bool same = p[0] == s && an == a && bn == b;
        s = p[0]; a = an; b = bn;
        if (same) break;
    }
    return score_serialised<B, JOINT>(ln, w, G, umax, s, a, b);
}

// the best of a group's candidates: smallest loss, the earliest of equals
__device__ __forceinline__ int best_of(const Fit *f, int n, int lane) {
    double loss = INFINITY;
    int idx = -1;
    for (int c = lane; c < n; c += 32) if (f[c].loss < loss) { loss = f[c].loss; idx = c; }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const double l2 = __shfl_xor_sync(0xffffffffu, loss, o);
        const int i2 = __shfl_xor_sync(0xffffffffu, idx, o);
        if (i2 >= 0 && (idx < 0 || l2 < loss || (l2 == loss && i2 < idx))) { loss = l2; idx = i2; }
    }
    return idx;   // -1: none is valid
}

template <int B>
__global__ void __launch_bounds__(SearchShape<B>::T) search_kernel(const float *__restrict__ W, const __grid_constant__ SearchPlan p,
                                                                   int8_t *__restrict__ k, float *__restrict__ scale,
                                                                   uint16_t *__restrict__ a, uint16_t *__restrict__ b) {
    using S = SearchShape<B>;
    constexpr int M = S::M, L = S::L, T = S::T;
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ double s_td[L], s_phi[3 * L], s_r127[128];
    __shared__ float s_tf[L], s_umax[32];
    __shared__ int s_next;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, NW = T / 32;
    const int G = p.G, GB = p.groups_per_block, ncand = p.n_int + p.n_shape;
    const int64_t g0 = (int64_t)blockIdx.x * GB;
    const int ngroups = (int)min((int64_t)GB, p.groups - g0);
    Weight *wt = reinterpret_cast<Weight *>(smem);                          // [GB][G + 1]
    Fit *fits = reinterpret_cast<Fit *>(wt + (size_t)GB * (G + 1));         // [2][GB][ncand + 1]; the last one: the continuous answer re-scored
    double *fin = reinterpret_cast<double *>(fits + (size_t)(p.dual ? 2 : 1) * GB * (ncand + 1));   // the last step's tables
    double *col = fin + S::FINAL / 8;
    Columns<B> ln;
    ln.z_ = col + tid; ln.zt_ = col + L * T + tid;
    ln.above = reinterpret_cast<float *>(col + 2 * L * T) + tid;
    ln.thr = reinterpret_cast<float *>(col) + tid;
    ln.carrier = reinterpret_cast<uint8_t *>(reinterpret_cast<float *>(col) + L * T) + tid;
    ln.a = 1.0; ln.b = 0.0;
    ln.td = s_td; ln.phi = s_phi; ln.tf = s_tf; ln.r127 = s_r127;

    for (int i = tid; i < L; i += T) {
        const double t = (double)i / (double)M, t2 = t * t, t3 = t2 * t;
        s_td[i] = t; s_tf[i] = __fdiv_rn((float)i, (float)M);
        s_phi[i] = t3; s_phi[L + i] = t - t3; s_phi[2 * L + i] = t2 - t3;
    }
    for (int i = tid; i < 128; i += T) s_r127[i] = (double)i / 127.0;
    if (tid == 0) s_next = 0;
    for (int gl = warp; gl < ngroups; gl += NW) {
        const float *w = W + (g0 + gl) * G;   // K is a multiple of G: group i of the matrix starts at i G
        float mx = 0.0f;
        for (int j = lane; j < G; j += 32) {
            Weight x;
            x.f = fabsf(w[j]); x.u = (double)x.f; x.pad = 0;
            wt[gl * (G + 1) + j] = x;
            if (x.f > mx) mx = x.f;
        }
        for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane == 0) s_umax[gl] = mx;
    }
    __syncthreads();

    // Chunks of 32 lanes of one kind, the long ones first: shapes (joint, continuous), clipped integers (joint, continuous).
    const int ch_shape = (ngroups * p.n_shape + 31) / 32, ch_int = (ngroups * p.n_int + 31) / 32;
    const int per_obj = p.dual ? 2 : 1, n_chunks = per_obj * (ch_shape + ch_int);
    for (;;) {
        int c = 0;
        if (lane == 0) c = atomicAdd(&s_next, 1);
        c = __shfl_sync(0xffffffffu, c, 0);
        if (c >= n_chunks) break;
        const bool shaped = c < per_obj * ch_shape;
        const int cc = shaped ? c : c - per_obj * ch_shape, ch = shaped ? ch_shape : ch_int, n = shaped ? p.n_shape : p.n_int;
        const bool joint = p.dual && cc < ch;
        const int item = (cc % ch) * 32 + lane;
        if (item < ngroups * n) {
            const int gl = item / n, cand = item % n;
            const float umax = s_umax[gl];
            if (umax != 0.0f) {
                double a0 = 1.0, b0 = 0.0, s0;
                int iters = 6, refine = 0;
                if (shaped) {
                    a0 = p.shapes[cand / p.clips][0]; b0 = p.shapes[cand / p.clips][1];
                    s0 = p.clip[cand % p.clips] * (double)umax;
                    iters = p.iters; refine = p.refine;
                } else {
                    const double clips_int[INT_CLIPS] = {1.0, 0.95, 0.9, 0.85, 0.8, 0.75, 0.7, 0.65, 0.6, 0.55, 0.5, 0.45, 0.4, 0.35, 0.3};
                    s0 = clips_int[cand] * (double)umax;
                }
                const Weight *w = wt + gl * (G + 1);
                Fit *out = fits + (size_t)((joint ? GB : 0) + gl) * (ncand + 1) + (shaped ? p.n_int : 0) + cand;
                *out = joint ? try_candidate<B, true>(ln, w, G, umax, a0, b0, s0, iters, refine)
                             : try_candidate<B, false>(ln, w, G, umax, a0, b0, s0, iters, refine);
            }
        }
        __syncwarp();
    }
    __syncthreads();

    // the best of each group, and the codes it stores
    for (int gl = warp; gl < ngroups; gl += NW) {
        const int64_t gi = g0 + gl;
        const float *w = W + gi * G;
        int8_t *out = k + gi * G;
        const float umax = s_umax[gl];
        if (umax == 0.0f) {   // all-zero group: s = 0, codes 0
            for (int j = lane; j < G; j += 32) out[j] = 0;
            if (lane == 0) { scale[gi] = 0.0f; a[gi] = 0x3C00; b[gi] = 0; }
            continue;
        }
        Fit *cont = fits + (size_t)gl * (ncand + 1);
        int win = best_of(cont, ncand, lane);
        Fit best;
        best.loss = INFINITY; best.s = umax; best.a16 = 0x3C00; best.b16 = 0;   // none valid: absmax integer quantisation
        if (win >= 0) best = cont[win];
        if (p.dual) {
            // The continuous fitter's answer competes too, re-scored under the joint objective and after the joint
            // candidates, so the dual-path result is never worse (jointly) than the continuous-only one.
            Fit *jf = cont + (size_t)GB * (ncand + 1);
            if (lane == 0) {
                jf[ncand].loss = INFINITY;
                if (win >= 0) jf[ncand] = try_candidate<B, true>(ln, wt + gl * (G + 1), G, umax, half_bits_to_double(best.a16), half_bits_to_double(best.b16), (double)best.s, 0, 0);
            }
            __syncwarp();
            win = best_of(jf, ncand + 1, lane);
            if (win >= 0) best = jf[win];
            else { best.s = umax; best.a16 = 0x3C00; best.b16 = 0; }
        }
        const bool joint = p.dual && win >= 0;
        const double sd = (double)best.s, av = half_bits_to_double(best.a16), bv = half_bits_to_double(best.b16);
        double *z = fin + (size_t)warp * 2 * L, *zt = z + L;   // joint: levels and carrier grid; else s z
        __syncwarp();
        for (int i = lane; i < L; i += 32) z[i] = joint ? level_curve(s_td[i], av, bv) : sd * level_curve(s_td[i], av, bv);
        if (joint) {
            const float af = (float)av, bf = (float)bv, c = __fsub_rn(__fsub_rn(1.0f, af), bf);
            for (int i = lane; i < L; i += 32) {
                const float t = s_tf[i];
                const float q = __fmul_rn(t, fmaf(t, fmaf(t, c, bf), af));
                zt[i] = s_r127[min(max(__float2int_rn(__fmul_rn(127.0f, q)), 0), 127)];
            }
        }
        __syncwarp();
        for (int j = lane; j < G; j += 32) {
            const double u = wt[gl * (G + 1) + j].u;
            const int i = joint ? joint_level(u, sd, z, zt, M) : nearest_level(u, z, M);
            out[j] = (int8_t)(w[j] < 0.0f ? -i : i);
        }
        if (lane == 0) { scale[gi] = best.s; a[gi] = best.a16; b[gi] = best.b16; }
        __syncwarp();
    }
}

// W1 (sign codes; s = mean |w| minimises sum (w - k s)^2) and effort 0 (symmetric absmax integer quantisation): one
// thread per group, nothing to search.
__global__ void __launch_bounds__(32) direct_kernel(const float *__restrict__ W, int B, int G, int64_t groups, int8_t *__restrict__ k,
                                                    float *__restrict__ scale, uint16_t *__restrict__ a, uint16_t *__restrict__ b) {
    const int64_t gi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= groups) return;
    const float *w = W + gi * G;
    int8_t *out = k + gi * G;
    double umax = 0.0, usum = 0.0;
    for (int j = 0; j < G; ++j) { const double u = fabs((double)w[j]); usum += u; if (u > umax) umax = u; }
    a[gi] = 0x3C00; b[gi] = 0;
    if (umax == 0.0) {
        scale[gi] = 0.0f;
        for (int j = 0; j < G; ++j) out[j] = (int8_t)(B == 1 ? 1 : 0);
        return;
    }
    if (B == 1) {
        scale[gi] = (float)(usum / G);
        for (int j = 0; j < G; ++j) out[j] = (int8_t)(w[j] >= 0.0f ? 1 : -1);
        return;
    }
    const int M = top_code(B);
    const float s_abs = (float)umax;
    double y[MAXL];
    for (int i = 0; i <= M; ++i) y[i] = (double)s_abs * level_curve((double)i / (double)M, 1.0, 0.0);
    for (int j = 0; j < G; ++j) {
        const int i = nearest_level(fabs((double)w[j]), y, M);
        out[j] = (int8_t)(w[j] < 0.0f ? -i : i);
    }
    scale[gi] = s_abs;
}

// Candidate shapes of the search (a deterministic set of monotone shapes; the uniform-integer point (1, 0) first).
// Effort 2: 4 x 3 shapes, 3 clips; 3: a dense grid, 6 clips.
int shape_list(int effort, double (*out)[2]) {
    int n = 0;
    out[n][0] = 1.0; out[n][1] = 0.0; ++n;
    if (effort == 2) {
        const double as[4] = {0.4, 0.6, 0.8, 1.0}, bs[3] = {-0.6, -0.3, 0.0};
        for (int i = 0; i < 4; ++i) for (int j = 0; j < 3; ++j) {
            if (as[i] == 1.0 && bs[j] == 0.0) continue;
            if (shape_margin(as[i], bs[j]) > 0.02) { out[n][0] = as[i]; out[n][1] = bs[j]; ++n; }
        }
        return n;
    }
    for (int i = 2; i <= 12; ++i) for (int j = -10; j <= 2; ++j) {
        const double a = 0.1 * i, b = 0.1 * j;
        if (i == 10 && j == 0) continue;
        if (shape_margin(a, b) > 0.02) { out[n][0] = a; out[n][1] = b; ++n; }
    }
    return n;
}

template <int B>
cudaError_t launch_search(const float *W, SearchPlan &p, int8_t *k, float *scale, uint16_t *a, uint16_t *b, cudaStream_t st) {
    using S = SearchShape<B>;
    // as many groups to a block as fill its warps several times over: more make the weights and results of a block too large
    const size_t per_group = (size_t)(p.G + 1) * sizeof(Weight) + (size_t)(p.dual ? 2 : 1) * (p.n_int + p.n_shape + 1) * sizeof(Fit);
    int gb = (int)((size_t)(32 * 1024) / per_group);
    gb = gb > 8 ? 8 : gb < 1 ? 1 : gb;
    p.groups_per_block = gb;
    const size_t smem = gb * per_group + (size_t)S::FINAL + (size_t)S::COL * S::T;
    static std::atomic<uint64_t> attr_done{0};
    cudaError_t e = ensure_func_attr(search_kernel<B>, attr_done, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
    if (e != cudaSuccess) return e;
    search_kernel<B><<<(unsigned)((p.groups + gb - 1) / gb), S::T, smem, st>>>(W, p, k, scale, a, b);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_encode_assign(const float *W, int B, int G, int64_t N, int64_t K, const float *scale, const uint16_t *a,
                                 const uint16_t *b, int joint, int8_t *k, cudaStream_t st) {
    const int64_t ng = K / G;
    assign_kernel<<<(unsigned)(N * ng), 128, 0, st>>>(W, B, G, K, ng, scale, a, b, joint && B > 2, k);
    return cudaGetLastError();
}
cudaError_t launch_encode_scale(const float *W, const int8_t *k, int B, int G, int64_t N, int64_t K, const uint16_t *a,
                                const uint16_t *b, int joint, float *scale, cudaStream_t st) {
    const int64_t ng = K / G;
    scale_kernel<<<(unsigned)(N * ng), 128, 0, st>>>(W, k, B, G, K, ng, a, b, joint && B > 2, scale);
    return cudaGetLastError();
}
cudaError_t launch_encode_losses(const float *W, const int8_t *k, int B, int G, int64_t N, int64_t K, const float *scale,
                                 const uint16_t *a, const uint16_t *b, double *LC, double *LA8, cudaStream_t st) {
    const int64_t ng = K / G;
    losses_kernel<<<(unsigned)(N * ng), 128, 0, st>>>(W, k, B, G, K, ng, scale, a, b, LC, LA8);
    return cudaGetLastError();
}
cudaError_t launch_encode_search(const float *W, int B, int G, int64_t N, int64_t K, int joint, int effort, int8_t *k,
                                 float *scale, uint16_t *a, uint16_t *b, cudaStream_t st) {
    const int64_t groups = N * (K / G);
    if (B == 1 || effort == 0) {
        direct_kernel<<<(unsigned)((groups + 31) / 32), 32, 0, st>>>(W, B, G, groups, k, scale, a, b);
        return cudaGetLastError();
    }
    static const double clips_fast[3] = {1.0, 0.85, 0.7}, clips_ref[6] = {1.0, 0.9, 0.8, 0.7, 0.6, 0.5};
    SearchPlan p;
    p.G = G; p.groups = groups;
    p.dual = joint && B > 2;   // W1 / W2 levels lie on the carrier grid: the objectives coincide
    p.n_int = INT_CLIPS;       // the clipped uniform-integer candidates always compete, and first: never worse than clipped INT
    p.clips = effort == 3 ? 6 : 3;
    for (int i = 0; i < p.clips; ++i) p.clip[i] = effort == 3 ? clips_ref[i] : clips_fast[i];
    p.iters = effort == 3 ? 4 : 3;
    p.refine = B == 2 ? 0 : effort == 3 ? 12 : 8;
    int shapes = effort >= 2 ? shape_list(effort, p.shapes) : 0;
    if (B == 2 && effort >= 2) shapes = 1;   // W2: the shape is not identifiable
    p.n_shape = shapes * p.clips;
    switch (B) {
        case 2: return launch_search<2>(W, p, k, scale, a, b, st);
        case 3: return launch_search<3>(W, p, k, scale, a, b, st);
        case 4: return launch_search<4>(W, p, k, scale, a, b, st);
        case 5: return launch_search<5>(W, p, k, scale, a, b, st);
        case 6: return launch_search<6>(W, p, k, scale, a, b, st);
        case 7: return launch_search<7>(W, p, k, scale, a, b, st);
        default: return launch_search<8>(W, p, k, scale, a, b, st);
    }
}

}  // namespace cq
