// fused.cuh -- the fused persistent trajectory kernel.
//
// One CTA evolves one trajectory at a time, through every step of its medium, and then fetches the
// next trajectory from a global work counter.  The wave function never leaves the SM: between the sine
// transforms it lives in registers (N/G values a thread), and shared memory only exchanges values
// between the threads inside a transform.
//
// One step (Sec. 3.3, steps 1-5) with T = T(tau_n) (Sec. 3.4, Bjorken):
//   x <- K_V(n) x        K_V = exp(-i V_eff dt/2) = static(c, l, r) * exp((er + i ei) T^3 r^2)
//   S = DST(x)           S_k = sum_j x_j sin(pi j k / N)
//   S <- K_T S           K_T = exp(-i T_kin(p_k) dt) * 2/N   (2/N = inverse DST scale)
//   x = DST(S)
//   x <- K_V(n) x, norm^2 = (L/N) sum |x_j|^2, jump if norm^2 <= r (Sec. 3.2.1, 3.4.3-3.4.4, 3.5)
// The end half-step of step n and the start half-step of step n+1 are applied as one factor
// static^2 * exp((er_n + er_{n+1}) r^2 + i (ei_n + ei_{n+1}) r^2); the norm after the end half-step is
// accumulated with the weights |K_V(n)|^2 = exp(2 er_n r^2) on the way.  On the rare steps that
// jump, the start half-step is turned into the new colour's and l's afterwards (all these factors are
// diagonal in r and commute with the jump's multiplication by r).
//
// The sine transform.  With X the length-2N FFT of the odd extension of x, X_k = -2i S_k, and both x and X
// are odd: only half of every pass is independent, and only that half is computed and stored.  Indices
// n = b + S m (m < R, S = 2N/R), k = kk + R q (kk < R):
//   first pass   Z_b[kk] = DFT_R of x_{b + S m} over m, for one b of every pair +-b (mod S);
//                A_kk[b] = W_2N^(b kk) Z_b[kk], and by the oddness A_{R-kk}[b] = -conj(W^(b kk))..., i.e.
//                A_kk[-b] = -W_2N^(-b kk) Z_b[R-kk]: one b fills the sequences kk = 1 .. R/2-1 at b and -b;
//   middle       FFT_S of each sequence over b = b1 + R m: DFT_M over m (in place), twiddle W_S^(b1 q1),
//   last pass    DFT_R over b1 -> X_{kk + R q1 + S q2}, q2 < R.
// The last pass leaves a thread with the points b + S q2, b = kk + R q1 -- the inputs of one first-pass
// butterfly of the next transform.  So the kinetic and potential factors and the norm act on registers
// between a last and a first pass, and a transform exchanges values through shared memory twice.
// (A transform through one N-point FFT with sine pre- and post-processing, which this replaced, needed
// four to five exchanges, a compensated prefix sum over the N/2 odd coefficients, and about 1.9 times the
// instructions; its running sum also carried the FFT's rounding errors along k.)
// The sequences kk = 0 (U, odd: U_{-q} = -U_q) and kk = R/2 (V, V_{-1-q} = -V_q) are half as long; they
// share one FFT_S of their sum P, and P_q + P_{-q} = V_q - V_{q-1} gives V by a prefix sum of S/2 values
// and U = P - V (split()).  The two sequences b = 0 and b = S/2 of the first pass (odd and half-odd in m)
// share the butterfly of slot 0 the same way, separated in closed form (special_in, special_mid).
// Which points a thread holds: fused_plan.h.
#pragma once
#include <type_traits>

#include "fused_launch.cuh"
#include "fused_plan.h"
#include "qtraj_device.cuh"

namespace qt {

// V selects the launch variant (fused_launch.cuh): 0, 1 the plan of the grid size with 512 or 640 resident
// threads per SM, 2 and 3 the radix-8 plans with 768 and 1024; 4 and 6 the traced twins of 0 and 2, 5 the
// KSU twin of 0, 7 the plain form's kernels (plain_step.cuh).
template <typename T, int N, int V = 0> struct FusedPlan {
    static constexpr PlanDims D = plan_dims(N, sizeof(T) == 8, V == 2 || V == 3 || V == 6 ? PLAN_RAD8 : V == 7 ? PLAN_PLAIN : PLAN_FUSED);
    static constexpr int R = D.R, E = D.E, M1 = D.M1, M2 = D.M2;
    static constexpr int H = R / 2;              // sequences
    static constexpr int M = M1 * M2;            // length of the middle transform
    static constexpr int S = R * M;              // length of a sequence
    static constexpr int G = N / E;              // threads per trajectory
    static constexpr int NS = E / R;             // slots per thread
    static constexpr int NSLOT = N / R;
    static constexpr bool TWL = plan_tw_last(D);
    // Shared-memory address of position b of a sequence: b + b/R (one pad element every R), so that the
    // stride-R accesses of the first and last passes are stride R+1 and conflict-free; the sequences are
    // SEQ apart, with SEQ = M (mod 16) where several sequences share a half-warp (M < 16), so that their
    // M-lane runs are adjacent modulo the banks.
    static constexpr int SEQ0 = S + S / R;
    static constexpr int SEQ = M < 16 ? SEQ0 + ((M - SEQ0) % 16 + 16) % 16 : SEQ0;
    static constexpr int BUF = H * SEQ;
    // butterflies a thread does in a middle pass, and the registers these take
    static constexpr int PER1 = (N / M1 + G - 1) / G, PER2 = (N / M2 + G - 1) / G;
    static constexpr int X0 = PER1 * M1 > E ? PER1 * M1 : E;
    static constexpr int XN = M2 > 1 && PER2 * M2 > X0 ? PER2 * M2 : X0;
    static_assert(N * 2 == R * R * M && G % R == 0 && M <= G && E % R == 0, "plan");
};

// ------------------------------------------------------------------------------------------------
// accumulators: FP32 forms accumulate sums of squares with compensated (cascaded) summation and
// combine partial sums in double-float (error-free transformations in FP32), so no FP64 instruction
// enters the step loop (GB300's FP64 pipe is narrow); FP64 forms accumulate in double.
// ------------------------------------------------------------------------------------------------
struct DF { float hi, lo; };

__device__ __forceinline__ DF two_sum(float a, float b)
{
    const float s = a + b, bb = s - a;
    return {s, (a - (s - bb)) + (b - bb)};
}
// commutative bit for bit (two_sum is exact; a.lo + b.lo is added first), so xor-butterfly
// reductions leave the same value in every lane
__device__ __forceinline__ DF df_add(DF a, DF b)
{
    DF s = two_sum(a.hi, b.hi);
    const float t = s.lo + (a.lo + b.lo);
    const float hi = s.hi + t;
    return {hi, t - (hi - s.hi)};
}

template <typename T> struct SqAcc;
template <> struct SqAcc<float> {
    DF v{0.f, 0.f};
    // v += w |a|^2 in plain FP32: a thread sums its E values in two chains (8 terms each at N = 4096), a
    // relative error of ~sqrt(8) x 6e-8 = 1.7e-7, random from step to step; the sums of the chains and
    // threads are then combined in double-float.  The norm feeds only the waiting-time comparison and the
    // jump's renormalisation, and the FP32 state's own norm is 0.4 .. 1.4e-6 off after 64 .. 300 steps, so
    // a compensated per-thread sum (as an earlier revision had) buys nothing the comparison can see.
    __device__ __forceinline__ void add_w(cpx<float> a, float w) { v.hi = fmaf(w, fmaf(a.x, a.x, a.y * a.y), v.hi); }
    __device__ __forceinline__ void shfl_add(unsigned mask, int off, int w)
    {
        DF o{__shfl_xor_sync(mask, v.hi, off, w), __shfl_xor_sync(mask, v.lo, off, w)};
        v = df_add(v, o);
    }
    __device__ __forceinline__ double value() const { return (double)v.hi + (double)v.lo; }
    __device__ __forceinline__ void merge(const SqAcc &o) { v = df_add(v, o.v); }
};
template <> struct SqAcc<double> {
    double v = 0.0;
    __device__ __forceinline__ void merge(const SqAcc &o) { v += o.v; }
    __device__ __forceinline__ void add_w(cpx<double> a, double w) { v = fma(w, fma(a.x, a.x, a.y * a.y), v); }
    __device__ __forceinline__ void shfl_add(unsigned mask, int off, int w) { v += __shfl_xor_sync(mask, v, off, w); }
    __device__ __forceinline__ double value() const { return v; }
};

template <int G> __device__ __forceinline__ unsigned lane_mask()
{
    return G >= 32 ? 0xffffffffu : ((1u << G) - 1u);
}

template <int G> __device__ __forceinline__ void traj_sync()
{
    if constexpr (G > 32) __syncthreads();
    else __syncwarp(lane_mask<G>());
}

// combines per-warp totals (equal in every lane of a warp) across the G threads of a trajectory in a
// fixed order; red holds >= G/32 doubles
template <int G> __device__ __forceinline__ double cross_warp(double v, double *red)
{
    if constexpr (G > 32) {
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
        __syncthreads();
        double s = 0.0;
#pragma unroll
        for (int w = 0; w < G / 32; ++w) s += red[w];
        __syncthreads();
        return s;
    } else {
        return v;
    }
}

// sum over the G threads of a trajectory (deterministic order, one value in every thread)
template <int G> __device__ __forceinline__ double slot_sum(double v, double *red)
{
    constexpr int W = G < 32 ? G : 32;
    const unsigned mask = lane_mask<G>();
#pragma unroll
    for (int off = W / 2; off > 0; off >>= 1) v += __shfl_xor_sync(mask, v, off, W);
    if constexpr (G <= 32) v = __shfl_sync(mask, v, 0, W);
    return cross_warp<G>(v, red);
}

// Eight sums over the G threads of a trajectory, left in fin[0..8) for the threads of its first warp.  The warp sums
// by halving -- each lane passes half of its values on and keeps the sums of the other half, 9 additions instead of
// 40 -- and the first eight lanes add the warps' sums: an FP64 addition takes a warp 64 cycles.  red holds >= 8 G/32
// doubles.
template <int G> __device__ __forceinline__ void slot_sums8(double (&v)[8], double *red, double *fin)
{
    constexpr int W = G < 32 ? G : 32, NW = G < 32 ? 1 : G / 32;
    const unsigned mask = lane_mask<G>();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int at = 0;   // the value this lane is left with
    if constexpr (W == 32) {
#pragma unroll
        for (int k = 4, off = 16; k > 0; k >>= 1, off >>= 1) {
            const bool up = lane & off;
#pragma unroll
            for (int i = 0; i < k; ++i) {
                const double mine = up ? v[i + k] : v[i], his = up ? v[i] : v[i + k];
                v[i] = mine + __shfl_xor_sync(mask, his, off, W);
            }
            at += up ? k : 0;
        }
#pragma unroll
        for (int off = 2; off > 0; off >>= 1) v[0] += __shfl_xor_sync(mask, v[0], off, W);
        if ((lane & 3) == 0) red[at * NW + warp] = v[0];
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
#pragma unroll
            for (int off = W / 2; off > 0; off >>= 1) v[i] += __shfl_xor_sync(mask, v[i], off, W);
            if (lane == 0) red[i] = v[i];
        }
    }
    traj_sync<G>();
    if (warp == 0) {
        for (int i = lane; i < 8; i += W) {
            double t = 0.0;
            for (int w = 0; w < NW; ++w) t += red[i * NW + w];
            fin[i] = t;
        }
        __syncwarp(mask);
    }
}

// A sum of products f u with a constant real f = h + l and FP32 complex u, both parts at once in packed FP32x2
// instructions: products and partial sums in error-free parts (the Dot2 scheme of Ogita, Rump and Oishi), some 2^-46
// of the terms' magnitudes.
struct Dot2 {
    float2 s = make_float2(0.f, 0.f), c = make_float2(0.f, 0.f);
    static __device__ __forceinline__ float2 neg(float2 a) { return make_float2(-a.x, -a.y); }
    __device__ __forceinline__ void add(float2 f, float2 u)   // f u, componentwise
    {
        const float2 p = __fmul2_rn(f, u), r = __ffma2_rn(f, u, neg(p));
        const float2 t = __fadd2_rn(s, p), b = __fadd2_rn(t, neg(s));
        const float2 e = __fadd2_rn(__fadd2_rn(s, neg(__fadd2_rn(t, neg(b)))), __fadd2_rn(p, neg(b)));
        c = __fadd2_rn(c, __fadd2_rn(e, r));
        s = t;
    }
    __device__ __forceinline__ void add(Prec<float>::Rl f, float2 u)
    {
        add(make_float2(f.h, f.h), u);
        c = __ffma2_rn(make_float2(f.l, f.l), u, c);
    }
    __device__ __forceinline__ double x() const { return (double)s.x + (double)c.x; }
    __device__ __forceinline__ double y() const { return (double)s.y + (double)c.y; }
};
// Where a norm's sum by Dot2 is taken: the parts of products below 2^-149 are lost and those above 2^128 overflow, N 2^-149
// in all, which is less than 2^-53 of a sum above 2^-80.  Other sums (states decayed without a jump, and non-finite
// ones), and states without a step behind them, whose overlaps may cancel to any depth, are taken again in FP64.
__device__ __forceinline__ bool dot2_holds(double norm) { return norm > 0x1p-80 && norm < 0x1p100; }
struct Dot1 {   // the FP64 form
    double s = 0.0, t = 0.0;
    __device__ __forceinline__ void add(double f, cpx<double> u) { s = fma(f, u.x, s); t = fma(f, u.y, t); }
    __device__ __forceinline__ void sq(cpx<double> u) { s = fma(u.x, u.x, s); t = fma(u.y, u.y, t); }
    __device__ __forceinline__ double x() const { return s; }
    __device__ __forceinline__ double y() const { return t; }
};

// squared norm over the G threads of a trajectory; FP32 forms reduce in double-float all the way and
// convert once, so no FP64 instruction is needed per thread beyond the final conversion
template <typename T, int G> __device__ __forceinline__ double slot_norm(SqAcc<T> acc, double *red)
{
    constexpr int W = G < 32 ? G : 32;
    const unsigned mask = lane_mask<G>();
#pragma unroll
    for (int off = W / 2; off > 0; off >>= 1) acc.shfl_add(mask, off, W);
    if constexpr (sizeof(T) == 4) {
        DF v = acc.v;
        if constexpr (G <= 32) {
            v.hi = __shfl_sync(mask, v.hi, 0, W);
            v.lo = __shfl_sync(mask, v.lo, 0, W);
        } else {
            DF *fr = reinterpret_cast<DF *>(red);
            if ((threadIdx.x & 31) == 0) fr[threadIdx.x >> 5] = v;
            __syncthreads();
            v = fr[0];
#pragma unroll
            for (int w = 1; w < G / 32; ++w) v = df_add(v, fr[w]);
            __syncthreads();
        }
        return (double)v.hi + (double)v.lo;
    } else {
        double v = acc.value();
        if constexpr (G <= 32) v = __shfl_sync(mask, v, 0, W);
        return cross_warp<G>(v, red);
    }
}

// The norm sum as the step loop compares it with the waiting-time threshold: double-float in the FP32
// forms (so that no FP64 instruction -- a slow pipe on GB300 -- runs in every step), double in FP64.
template <typename T> struct NormSum { using type = double; };
template <> struct NormSum<float> { using type = DF; };

template <typename T, int G> __device__ __forceinline__ typename NormSum<T>::type slot_norm_sum(SqAcc<T> acc, double *red)
{
    if constexpr (sizeof(T) == 4) {
        constexpr int W = G < 32 ? G : 32;
        const unsigned mask = lane_mask<G>();
#pragma unroll
        for (int off = W / 2; off > 0; off >>= 1) acc.shfl_add(mask, off, W);
        DF v = acc.v;
        if constexpr (G <= 32) {
            v.hi = __shfl_sync(mask, v.hi, 0, W);
            v.lo = __shfl_sync(mask, v.lo, 0, W);
        } else {
            DF *fr = reinterpret_cast<DF *>(red);
            if ((threadIdx.x & 31) == 0) fr[threadIdx.x >> 5] = v;
            __syncthreads();
            v = fr[0];
#pragma unroll
            for (int w = 1; w < G / 32; ++w) v = df_add(v, fr[w]);
            __syncthreads();
        }
        return v;
    } else {
        return slot_norm<T, G>(acc, red);
    }
}

// the step loop's norm sum: as slot_norm_sum, with one barrier, which also tells that every thread has read
// the transform's output (redh is written again only several barriers later)
template <typename T, int G> __device__ __forceinline__ typename NormSum<T>::type step_norm(SqAcc<T> acc, typename NormSum<T>::type *redh)
{
    if constexpr (G <= 32) {
        const typename NormSum<T>::type v = slot_norm_sum<T, G>(acc, nullptr);
        __syncwarp(lane_mask<G>());
        return v;
    } else {
        const unsigned mask = lane_mask<G>();
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) acc.shfl_add(mask, off, 32);
        if ((threadIdx.x & 31) == 0) redh[threadIdx.x >> 5] = acc.v;
        __syncthreads();
        acc.v = redh[0];
#pragma unroll
        for (int w = 1; w < G / 32; ++w) {
            SqAcc<T> o;
            o.v = redh[w];
            acc.merge(o);
        }
        return acc.v;
    }
}

// The waiting-time threshold in the form of the norm sum it is compared with: r / dr (the norm is
// dr times the sum), as a normalised double-float in FP32 forms, computed in FP64 once per waiting
// period.  The comparisons are then exact on the double-float values.
template <typename T> struct Threshold;
template <> struct Threshold<double> {
    double thr, dr;
    __device__ void set(double r, double dr_) { thr = r; dr = dr_; }
    __device__ bool finite(double s) const { return isfinite(s * dr); }
    __device__ bool reached(double s) const { return s * dr <= thr; }
    __device__ bool near(double s, double eps) const { return fabs(s * dr - thr) < eps; }
};
template <> struct Threshold<float> {
    DF t;
    float eps_s;
    __device__ void set(double r, double dr)
    {
        const double q = r / dr;
        t.hi = (float)q;
        t.lo = (float)(q - (double)t.hi);
        eps_s = (float)(border_eps<float>() / dr);
    }
    __device__ bool finite(DF s) const { return isfinite(s.hi) && isfinite(s.lo); }
    __device__ bool reached(DF s) const { return s.hi < t.hi || (s.hi == t.hi && s.lo <= t.lo); }
    __device__ bool near(DF s, double) const { return fabsf((s.hi - t.hi) + (s.lo - t.lo)) < eps_s; }
};

// exp(x) and (cos, sin)(pi y): the pi-scaled form has no large-argument reduction path
__device__ __forceinline__ float k_exp(float x) { return expf(x); }
__device__ __forceinline__ double k_exp(double x) { return exp(x); }

template <typename T> __device__ __noinline__ T table_T3_far(const double *p, int len, T tau, int *seg)
{
    int s = *seg;
    const T v = table_T3<T>(p, len, tau, s);
    *seg = s;
    return v;
}

// f1 = exp(a) exp(i pi y) - 1, the deviation from 1 of a dynamic factor, for a <= 0 (also returns
// exp(a) - 1).
// FP32: truncated Taylor series at 0 -- exp(a) - 1 to degree 8 for a >= -1/2 (truncation below
// |a|^9/9! <= 5.4e-9), sin(t) to degree 9 and cos(t) - 1 to degree 10 in t = pi y for |t| <= 1
// (truncation below 2.8e-8 and 2.1e-9) -- each accurate relative to the small quantity it returns;
// outside those ranges (large r, where |f1| is no longer small) the library functions.
// FP64: exp and sincospi; a rounding next to 1 is 1e-16 there and does not matter.
template <typename T> struct Dyn;
// the rare points outside the series' ranges, kept out of line so the hot loop stays small
static __device__ __noinline__ void dyn_far(float a, float y, float *em1, float *s, float *cm1)
{
    *em1 = expf(a) - 1.0f;
    float sh, ch;
    sincospif(0.5f * y, &sh, &ch);
    *s = 2.0f * sh * ch;
    *cm1 = -2.0f * sh * sh;
}

template <> struct Dyn<float> {
    static __device__ __forceinline__ void f1(float a, float y, float *fr, float *fi, float *e)
    {
        f1t(a, 3.14159265358979f * y, fr, fi, e);
    }
    // f1 from the phase t = pi y (the hot loop forms t directly; beyond the series' range y is
    // recomputed from t)
    static __device__ __forceinline__ void f1t(float a, float t, float *fr, float *fi, float *e)
    {
        float em1, s, cm1;
        if (a >= -0.5f && fabsf(t) <= 1.0f) {
            float p = 1.0f / 40320.0f;
            p = fmaf(p, a, 1.0f / 5040.0f);
            p = fmaf(p, a, 1.0f / 720.0f);
            p = fmaf(p, a, 1.0f / 120.0f);
            p = fmaf(p, a, 1.0f / 24.0f);
            p = fmaf(p, a, 1.0f / 6.0f);
            p = fmaf(p, a, 0.5f);
            p = fmaf(p, a, 1.0f);
            em1 = a * p;
            const float u = t * t;
            float ps = 1.0f / 362880.0f;
            ps = fmaf(ps, u, -1.0f / 5040.0f);
            ps = fmaf(ps, u, 1.0f / 120.0f);
            ps = fmaf(ps, u, -1.0f / 6.0f);
            ps = fmaf(ps, u, 1.0f);
            s = t * ps;
            float pc = -1.0f / 3628800.0f;
            pc = fmaf(pc, u, 1.0f / 40320.0f);
            pc = fmaf(pc, u, -1.0f / 720.0f);
            pc = fmaf(pc, u, 1.0f / 24.0f);
            pc = fmaf(pc, u, -0.5f);
            cm1 = u * pc;
        } else {
            dyn_far(a, t * 0.318309886183790672f, &em1, &s, &cm1);
        }
        const float mag = 1.0f + em1;
        *fr = fmaf(cm1, mag, em1);
        *fi = s * mag;
        *e = em1;
    }
    // both points of a pair at once in packed FP32x2 instructions, the same operations per component
    // as f1t (bit-identical), for arguments in the series' range
    static __device__ __forceinline__ float2 rep(float v) { return make_float2(v, v); }
    static __device__ __forceinline__ float2 em1_2(float2 a)
    {
        float2 p = __ffma2_rn(rep(1.0f / 40320.0f), a, rep(1.0f / 5040.0f));
        p = __ffma2_rn(p, a, rep(1.0f / 720.0f));
        p = __ffma2_rn(p, a, rep(1.0f / 120.0f));
        p = __ffma2_rn(p, a, rep(1.0f / 24.0f));
        p = __ffma2_rn(p, a, rep(1.0f / 6.0f));
        p = __ffma2_rn(p, a, rep(0.5f));
        p = __ffma2_rn(p, a, rep(1.0f));
        return __fmul2_rn(a, p);
    }
    static __device__ __forceinline__ void sc2(float2 t, float2 *s, float2 *cm1)   // sin(t), cos(t) - 1
    {
        const float2 u = __fmul2_rn(t, t);
        float2 ps = __ffma2_rn(rep(1.0f / 362880.0f), u, rep(-1.0f / 5040.0f));
        ps = __ffma2_rn(ps, u, rep(1.0f / 120.0f));
        ps = __ffma2_rn(ps, u, rep(-1.0f / 6.0f));
        ps = __ffma2_rn(ps, u, rep(1.0f));
        *s = __fmul2_rn(t, ps);
        float2 pc = __ffma2_rn(rep(-1.0f / 3628800.0f), u, rep(1.0f / 40320.0f));
        pc = __ffma2_rn(pc, u, rep(-1.0f / 720.0f));
        pc = __ffma2_rn(pc, u, rep(1.0f / 24.0f));
        pc = __ffma2_rn(pc, u, rep(-0.5f));
        *cm1 = __fmul2_rn(u, pc);
    }
    static __device__ __forceinline__ void f1t2(float2 a, float2 t, float2 *fr, float2 *fi, float2 *e)
    {
        const float2 em1 = em1_2(a);
        float2 s, cm1;
        sc2(t, &s, &cm1);
        const float2 mag = __fadd2_rn(rep(1.0f), em1);
        *fr = __ffma2_rn(cm1, mag, em1);
        *fi = __fmul2_rn(s, mag);
        *e = em1;
    }
    // the same beyond the series' range, reduced to it by Cody and Waite's two-part constants: exp(a) = 2^n exp(a - n ln 2), and t - 2 pi k quartered
    // and doubled back twice (cos 2x - 1 = -2 sin^2 x, sin 2x = 2 sin x (1 + (cos x - 1))); a < -87 counts as
    // -87 (not a NaN, which 0 x inf at r = 0 is and which the norm has to show), |t| <= 1e5
    static __device__ __forceinline__ void far2(float2 a, float2 t, float2 *fr, float2 *fi, float2 *e)
    {
        const float2 magic = rep(12582912.0f);   // 1.5 x 2^23: adding it rounds to the nearest integer
        a = make_float2(a.x < -87.0f ? -87.0f : a.x, a.y < -87.0f ? -87.0f : a.y);
        const float2 nm = __ffma2_rn(a, rep(1.44269504088896341f), magic);
        const float2 n = __fadd2_rn(nm, rep(-12582912.0f));
        float2 r = __ffma2_rn(n, rep(-0.693147182464599609f), a);
        r = __ffma2_rn(n, rep(1.90465429995776804e-9f), r);
        const float2 sc = make_float2(__int_as_float((__float_as_int(nm.x) << 23) + 0x3f800000),
                                      __int_as_float((__float_as_int(nm.y) << 23) + 0x3f800000));   // 2^n
        const float2 em1 = __ffma2_rn(sc, em1_2(r), __fadd2_rn(sc, rep(-1.0f)));
        const float2 k = __fadd2_rn(__ffma2_rn(t, rep(0.159154943091895336f), magic), rep(-12582912.0f));
        t = __ffma2_rn(k, rep(-6.28318548202514648f), t);
        t = __ffma2_rn(k, rep(1.74845560e-7f), t);
        float2 s, c;
        sc2(__fmul2_rn(t, rep(0.25f)), &s, &c);
        float2 s2 = __fmul2_rn(s, rep(2.0f)), c2 = __fmul2_rn(s2, make_float2(-s.x, -s.y));
        s2 = __ffma2_rn(s2, c, s2);
        s = __fmul2_rn(s2, rep(2.0f));
        c = __fmul2_rn(s, make_float2(-s2.x, -s2.y));
        s = __ffma2_rn(s, c2, s);
        const float2 mag = __fadd2_rn(rep(1.0f), em1);
        *fr = __ffma2_rn(c, mag, em1);
        *fi = __fmul2_rn(s, mag);
        *e = em1;
    }
};
template <> struct Dyn<double> {
    // exp(a + i t) and m = exp(a); Taylor series where both parts are small (truncation below 2^-55)
    template <bool PHASE> static __device__ __forceinline__ cpx<double> cexp(double a, double t, double *m)
    {
        double s = 0.0, c = 1.0, e;
        if (fabs(a) <= 0.125 && (!PHASE || fabs(t) <= 0.125)) {
            e = 1.0 / 39916800.0;
            e = fma(e, a, 1.0 / 3628800.0);
            e = fma(e, a, 1.0 / 362880.0);
            e = fma(e, a, 1.0 / 40320.0);
            e = fma(e, a, 1.0 / 5040.0);
            e = fma(e, a, 1.0 / 720.0);
            e = fma(e, a, 1.0 / 120.0);
            e = fma(e, a, 1.0 / 24.0);
            e = fma(e, a, 1.0 / 6.0);
            e = fma(e, a, 0.5);
            e = fma(e, a, 1.0);
            e = fma(e, a, 1.0);
            if (PHASE) {
                const double u = t * t;
                s = fma(fma(fma(fma(1.0 / 362880.0, u, -1.0 / 5040.0), u, 1.0 / 120.0), u, -1.0 / 6.0), u, 1.0) * t;
                c = fma(fma(fma(fma(fma(-1.0 / 3628800.0, u, 1.0 / 40320.0), u, -1.0 / 720.0), u, 1.0 / 24.0), u, -0.5), u, 1.0);
            }
        } else {
            e = exp(a);
            if (PHASE) sincospi(t * 0.318309886183790671537767526745, &s, &c);
        }
        *m = e;
        return PHASE ? mk(e * c, e * s) : mk(e, 0.0);
    }
    // exp(z) for the temperature's change over one step (factor_regs): the series to z^3
    static __device__ __forceinline__ double near1(double z) { return 1.0 + z * (1.0 + z * (0.5 + z * (1.0 / 6.0))); }
    static __device__ __forceinline__ void f1(double a, double y, double *fr, double *fi, double *e)
    {
        const double mag = exp(a);
        double s, c;
        sincospi(y, &s, &c);
        *fr = mag * c - 1.0;
        *fi = mag * s;
        *e = mag - 1.0;
    }
};
__device__ __forceinline__ void k_sincospi(float y, float *s, float *c) { sincospif(y, s, c); }
__device__ __forceinline__ void k_sincospi(double y, double *s, double *c) { sincospi(y, s, c); }

// static factor of a (colour, l) row beyond the table (l >= LTAB, some 33,000 jumps from l = 0),
// evaluated in FP64; span 1 = half step, 2 = full step
template <typename T>
__device__ __noinline__ typename Prec<T>::S static_far(double coul, double M, double dt, int l, double r, double span)
{
    const double V = coul / r + (double)l * (l + 1) / (M * r * r);
    double s, c;
    sincos(-V * dt * 0.5 * span, &s, &c);
    return Prec<T>::make_s(c, s);
}

// ------------------------------------------------------------------------------------------------
// the isotropic KSU potential (App. E): per-step scalars at one temperature and the per-point
// dynamic part V_R + a/r (the Cornell -a/r sits in the static factor) and V_I
// ------------------------------------------------------------------------------------------------
template <typename T> struct KsuT {
    T m;      // Debye mass m_D(T)
    T two_s;  // 2 sigma / m_D
    T gI;     // alpha_s(2 pi T) C_F T: V_I = -gI phi(m_D r)
};

__device__ __forceinline__ float k_log(float x) { return logf(x); }
__device__ __forceinline__ double k_log(double x) { return log(x); }
__device__ __forceinline__ float k_cbrt(float x) { return cbrtf(x); }
__device__ __forceinline__ double k_cbrt(double x) { return cbrt(x); }

template <typename T> __device__ __forceinline__ KsuT<T> ksu_at(const Tables<T> &tb, T T3)
{
    const T Tt = k_cbrt(T3);
    const T mu = (T)6.28318530717958647692 * Tt;
    const T as = tb.ksu_alpha0 / ((T)1 + tb.ksu_alpha0 * tb.ksu_b0 * k_log(mu * mu / tb.ksu_mu0sq));
    const T m = Tt * sqrt(tb.ksu_md2 * as);
    return {m, tb.ksu_two_sigma / m, as * tb.ksu_cf * Tt};
}

// phi(x) of V_I: the small-argument series below KSU_PHI_A0, cubic Hermite interpolation of the
// table up to KSU_PHI_A1, the asymptotic series 1 - sum_j (2j)! (2j+2) / x^(2j+2) above
template <typename T> __device__ __forceinline__ T ksu_phi(const Tables<T> &tb, T x)
{
    if (x < (T)KSU_PHI_A0) {
        const T y = x * x;
        T pl = (T)0, pc = (T)0;
#pragma unroll
        for (int k = KSU_PHI_SER - 1; k >= 0; --k) {
            pl = (pl + tb.phi_ser[2 * k]) * y;
            pc = (pc + tb.phi_ser[2 * k + 1]) * y;
        }
        return x > (T)0 ? -(pl * k_log(x) + pc) : (T)0;
    }
    if (x < (T)KSU_PHI_A1) {
        const T u = (x - (T)KSU_PHI_A0) * (T)KSU_PHI_PER;
        int i = (int)u;
        if (i > KSU_PHI_NODES - 2) i = KSU_PHI_NODES - 2;
        const T s = u - (T)i, s2 = s * s, s3 = s2 * s;
        const T *n = tb.phi_tab + 2 * i;
        const T h00 = (T)2 * s3 - (T)3 * s2 + (T)1, h10 = s3 - (T)2 * s2 + s, h01 = (T)3 * s2 - (T)2 * s3, h11 = s3 - s2;
        return h00 * n[0] + h10 * n[1] + h01 * n[2] + h11 * n[3];
    }
    const T q = (T)1 / (x * x);
    T p = (T)6706022400.0;
    p = fma(p, q, (T)43545600.0);
    p = fma(p, q, (T)403200.0);
    p = fma(p, q, (T)5760.0);
    p = fma(p, q, (T)144.0);
    p = fma(p, q, (T)8.0);
    p = fma(p, q, (T)2.0);
    return (T)1 - p * q;
}

// at grid point j > 0 and one temperature: vd = V_R + a/r (V_R = min(KMS, V_vac(r_SB))) and vi = V_I
template <typename T> __device__ __forceinline__ void ksu_point(const Tables<T> &tb, const KsuT<T> &k, T fj, T &vd, T &vi)
{
    const T aor = tb.ksu_a_dr / fj, r_sig = tb.ksu_sig_dr * fj;     // a/r, sigma r
    const T x = k.m * (fj * (T)tb.dr);
    const T e = exp(-x);
    // 1 - (1 + x) e^-x, by its series below 0.05 (the difference cancels there)
    T g;
    if (x < (T)0.05) {
        T p = (T)(-1.0 / 3991680.0);              // the terms (-1)^n (n-1) x^n / n!, n = 2 .. 11
        p = fma(p, x, (T)(1.0 / 403200.0));
        p = fma(p, x, (T)(-1.0 / 45360.0));
        p = fma(p, x, (T)(1.0 / 5760.0));
        p = fma(p, x, (T)(-1.0 / 840.0));
        p = fma(p, x, (T)(1.0 / 144.0));
        p = fma(p, x, (T)(-1.0 / 30.0));
        p = fma(p, x, (T)(1.0 / 8.0));
        p = fma(p, x, (T)(-1.0 / 3.0));
        p = fma(p, x, (T)0.5);
        g = p * x * x;
    } else {
        g = (T)1 - ((T)1 + x) * e;
    }
    vd = aor * g + k.two_s * ((T)1 - e) - r_sig * e;   // KMS + a/r
    if (vd - aor > tb.ksu_cap) vd = tb.ksu_cap + aor;  // the string-breaking cap
    vi = -k.gI * ksu_phi(tb, x);
}

// in-place DFT of RR values (natural order in); output k lands in slot operm(k).  HL: the FP32 constants in hi + lo
// parts (the KSU kernel), else as directions (Prec<float>::D)
template <typename T, int RR, bool HL = false> struct DFTI {
    static __device__ __forceinline__ cpx<T> tw(cpx<T> a, int j) { return HL ? tw16<T>(a, j) : tw32<T>(a, 2 * j); }
    static __device__ __forceinline__ constexpr int operm(int k)
    {
        if constexpr (RR == 32) return (k % 4) * 8 + DFTI<T, 8, HL>::operm(k / 4);
        else if constexpr (RR == 16) return (k % 4) * 4 + k / 4;
        else if constexpr (RR == 8) return (k % 4) * 2 + k / 4;
        else return k;
    }
    static __device__ __forceinline__ void run(cpx<T> *x)
    {
        if constexpr (RR == 32) {
#pragma unroll
            for (int n2 = 0; n2 < 8; ++n2) {
                dft4(x[n2], x[8 + n2], x[16 + n2], x[24 + n2]);      // k1 of column n2 at slot n2 + 8 k1
                x[8 + n2] = tw32<T>(x[8 + n2], n2 * 1);
                x[16 + n2] = tw32<T>(x[16 + n2], n2 * 2);
                x[24 + n2] = tw32<T>(x[24 + n2], n2 * 3);
            }
#pragma unroll
            for (int k1 = 0; k1 < 4; ++k1) DFTI<T, 8, HL>::run(x + 8 * k1);
        } else if constexpr (RR == 16) {
#pragma unroll
            for (int n2 = 0; n2 < 4; ++n2) {
                dft4(x[n2], x[4 + n2], x[8 + n2], x[12 + n2]);       // k1 of column n2 at slot n2 + 4 k1
                x[4 + n2] = tw(x[4 + n2], n2 * 1);
                x[8 + n2] = tw(x[8 + n2], n2 * 2);
                x[12 + n2] = tw(x[12 + n2], n2 * 3);
            }
#pragma unroll
            for (int k1 = 0; k1 < 4; ++k1) dft4(x[4 * k1], x[4 * k1 + 1], x[4 * k1 + 2], x[4 * k1 + 3]);
        } else if constexpr (RR == 8) {
#pragma unroll
            for (int n2 = 0; n2 < 2; ++n2) {
                dft4(x[n2], x[2 + n2], x[4 + n2], x[6 + n2]);        // k1 of column n2 at slot n2 + 2 k1
                x[2 + n2] = tw(x[2 + n2], 2 * n2 * 1);
                x[4 + n2] = tw(x[4 + n2], 2 * n2 * 2);
                x[6 + n2] = tw(x[6 + n2], 2 * n2 * 3);
            }
#pragma unroll
            for (int k1 = 0; k1 < 4; ++k1) dft2(x[2 * k1], x[2 * k1 + 1]);
        } else if constexpr (RR == 4) {
            dft4(x[0], x[1], x[2], x[3]);
        } else if constexpr (RR == 2) {
            dft2(x[0], x[1]);
        }
    }
};

// ------------------------------------------------------------------------------------------------
// the sine transform
// ------------------------------------------------------------------------------------------------
template <typename T, int N, int V> struct Sine {
    using P = FusedPlan<T, N, V>;
    using PR = Prec<T>;
    using C = typename Prec<T>::C;
    static constexpr int R = P::R, H = P::H, G = P::G, M = P::M, S = P::S, NS = P::NS, SEQ = P::SEQ;
    // (the products stay scalar: as packed FP32x2 instructions, with their operands regrouped, hi+lo products ran 8%
    // slower at N = 8192 and 4% at 16384)
    using D = typename Prec<T>::D;
    using DR = DFTI<T, R>;
    static __device__ __forceinline__ cpx<T> cmul(cpx<T> x, D w) { return PR::muld(x, w); }
    static __device__ __forceinline__ cpx<T> neg(cpx<T> a) { return mk(-a.x, -a.y); }

    // addresses of position b of a sequence and of its mirror S - b
    static __device__ __forceinline__ int pos(int b) { return b + b / R; }

    // Slot 0 holds y_m = x_{S m} (m < R/2) and w_m = x_{S/2 + S m} (m >= R/2), the independent halves of the
    // odd sequence y (y_0 = y_{R/2} = 0, y_{R-m} = -y_m) and of w (w_{R-1-m} = -w_m): y + w, in place
    static __device__ __forceinline__ void special_in(cpx<T> *r)
    {
        r[0] = neg(r[R - 1]);
#pragma unroll
        for (int m = 1; m < H; ++m) {
            r[R - m] = r[R - m] - r[m];
            r[m] = r[m] - r[R - 1 - m];
        }
    }

    // The DFT Z of y + w is left at the positions 0 (Z[k]) and S/2 (Z[R-k]) of sequence k, and the threads of
    // the middle pass that read both separate them: y's part is odd in k and w's obeys Z_w[-k] = -W_R^k
    // Z_w[k], so Z_w[k] = (Z[k] + Z[-k]) / (1 - W_R^k) (at most 1/(2 sin(pi/R)) times the sum), and with w's
    // first-pass twiddle W_2R^k and q = Z[k] + Z[-k], d = Z[k] - Z[-k]:
    // A_k[S/2] = -i q / (2 sin(pi k/R)), A_k[0] = d/2 + (i/2) cot(pi k/R) q.
    static __device__ __forceinline__ void special_out(const cpx<T> *x, cpx<T> *buf)
    {
        constexpr int p2 = S / 2 + S / 2 / R;
#pragma unroll
        for (int k = 1; k < H; ++k) {
            buf[k * SEQ] = x[DR::operm(k)];
            buf[k * SEQ + p2] = x[DR::operm(R - k)];
        }
        buf[0] = mk<T>(0, 0);
        buf[p2] = mul_mi(x[DR::operm(H)]);
    }
    static __device__ __forceinline__ void special_mid(cpx<T> &a, cpx<T> &b, const C *ts, int k)
    {
        const C w = PR::ld(ts + k);   // (1 / (2 sin), cot / 2)
        const cpx<T> q = a + b, d = scale(a - b, (T)0.5), al = PR::mulr(q, PR::re(w)), be = PR::mulr(q, PR::im(w));
        a = d + mul_i(be);
        b = mul_mi(al);
    }

    // First pass: the slots' DFTs, twiddles, and the writes of every sequence at b and -b.  pb, pm: the
    // addresses of b and S - b of the thread's slots.
    static __device__ __forceinline__ void first(cpx<T> *x, cpx<T> *buf, const D *ta, const C *tha, int g,
                                                 const int *pb, const int *pm)
    {
        if (g == 0) special_in(x);
#pragma unroll
        for (int t = 0; t < NS; ++t) {
            cpx<T> *v = x + t * R;
            DR::run(v);
            if (t == 0 && g == 0) {
                special_out(v, buf);
            } else {
                const D *w = ta + g + t * G;
                cpx<T> *ob = buf + pb[t], *om = buf + pm[t];
#pragma unroll
                for (int k = 1; k < H; ++k) {
                    const D wk = PR::ldd(w + (k - 1) * P::NSLOT);
                    ob[k * SEQ] = cmul(v[DR::operm(k)], wk);
                    om[k * SEQ] = cmul(v[DR::operm(R - k)], PR::ncj(wk));
                }
                // the sequence P = U + V at b: u + th z, at -b: -u - conj(th) z, th = e^(-i pi b/S)
                const C th = PR::ld(tha + g + t * G);
                const cpx<T> u = v[0], z = v[DR::operm(H)];
                const cpx<T> s = PR::mulr(z, PR::re(th)), d = PR::mulr(z, PR::im(th));
                const cpx<T> a = u + s, b = mul_i(d);
                ob[0] = a + b;
                om[0] = b - a;
            }
        }
    }

    // One middle pass of radix RM in place: butterfly i = (kk RO + o) R + b1 of the values at
    // b1 + R (LO o + LM m), m < RM.  TW 0: none, 1: the last pass's twiddle W_S^(b1 q1) from tm [q1][b1]
    // (M2 = 1), 2: the inner twiddle W_M^(m2 k1) from ti [k1][m2] (o = m2).
    template <int RM, int RO, int LO, int LM, int TW, bool FIRST>
    static __device__ __forceinline__ void mid_pass(cpx<T> *x, cpx<T> *buf, const D *tw, const C *ts, int g)
    {
        constexpr int NB = N / RM, PER = (NB + G - 1) / G;
        const int b1 = g % R;   // the same for all of a thread's butterflies (R divides G)
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const int i = g + q * G;
            if (NB % G == 0 || i < NB) {
                const int o = i / R % RO, kk = i / (R * RO);
                const cpx<T> *p = buf + kk * SEQ + b1 + (R + 1) * LO * o;
#pragma unroll
                for (int m = 0; m < RM; ++m) x[q * RM + m] = p[(R + 1) * LM * m];
                // the positions 0 and S/2 (both at o = 0: M1 is even)
                if (FIRST && b1 == 0 && o == 0 && kk > 0) special_mid(x[q * RM], x[q * RM + RM / 2], ts, kk);
                DFTI<T, RM>::run(x + q * RM);
            }
        }
#pragma unroll
        for (int m = 0; m < RM; ++m) {
            D w{};
            if (m && TW == 1) w = PR::ldd(tw + m * R + b1);
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                const int i = g + q * G;
                if (NB % G == 0 || i < NB) {
                    const int o = i / R % RO, kk = i / (R * RO);
                    if (m && TW == 2) w = PR::ldd(tw + m * RO + o);
                    cpx<T> v = x[q * RM + DFTI<T, RM>::operm(m)];
                    if (m && TW) v = cmul(v, w);
                    buf[kk * SEQ + b1 + (R + 1) * (LO * o + LM * m)] = v;
                }
            }
        }
    }

    static __device__ __forceinline__ void mid(cpx<T> *x, cpx<T> *buf, const D *tm, const D *ti, const C *ts, int g)
    {
        if constexpr (P::M2 == 1) {
            mid_pass<P::M1, 1, 0, 1, P::TWL ? 0 : 1, true>(x, buf, tm, ts, g);
        } else {
            // m = m2 + M2 m1: DFT over m1 -> k1, twiddle, DFT over m2 -> k2; q1 = k1 + M1 k2 at M2 k1 + k2
            mid_pass<P::M1, P::M2, 1, P::M2, 2, true>(x, buf, ti, ts, g);
            traj_sync<G>();
            mid_pass<P::M2, P::M1, P::M2, 1, 0, false>(x, buf, nullptr, nullptr, g);
        }
    }

    // Last pass: X_{b + S q2} into value q2 of every slot (natural order)
    static __device__ __forceinline__ void last(cpx<T> *x, cpx<T> *buf, const D *tm, int g)
    {
        constexpr bool SAME = G % M == 0;   // a thread's slots share q1
        cpx<T> y[NS * R];
#pragma unroll
        for (int b1 = 0; b1 < R; ++b1) {
            D w{};
            if (P::TWL && SAME && b1) w = PR::ldd(tm + b1 * M + g % M);
#pragma unroll
            for (int t = 0; t < NS; ++t) {
                const int s = g + t * G, q1 = s % M;
                const int loc = P::M2 == 1 ? q1 : q1 / P::M1 + P::M2 * (q1 % P::M1);
                cpx<T> v = buf[s / M * SEQ + (R + 1) * loc + b1];
                if (P::TWL && b1) {
                    if (!SAME) w = PR::ldd(tm + b1 * M + q1);
                    v = cmul(v, w);
                }
                y[t * R + b1] = v;
            }
        }
#pragma unroll
        for (int t = 0; t < NS; ++t) {
            DR::run(y + t * R);
#pragma unroll
            for (int m = 0; m < R; ++m) x[t * R + m] = y[t * R + DR::operm(m)];
        }
        if constexpr (M > 32) traj_sync<G>();
        if (M > 32 || g < 32) split(x, buf, g);   // (warp 0)
    }

    // The kk = 0 slots (threads g < M) hold P_q = U_q + V_q, q = g + M m; leaves V_q in the slots g >= M/2,
    // U_q in those below, and slot 0's two half sequences (special_in).  V_q = P_0 + sum_{i=1..q} (P_i +
    // P_{-i}) for q < S/2, through the kk = 0 sequence's own shared memory: each of LN lanes of warp 0 sums a run of
    // CH values, the runs' totals are scanned with shuffles, and V overwrites P's lower half (only the run's
    // owner reads it; the upper half stays).  The sum carries the rounding errors of at most S/2 values of
    // 2/R of the spectrum, both ends tied down.  For M > 32 (radix-8 variants) warp 0 sums for all and every thread calls this.
    static __device__ __forceinline__ void split(cpx<T> *x, cpx<T> *buf, int g)
    {
        constexpr int LN = G < 32 ? G : 32, CH = S / 2 / LN;
        static_assert(CH * LN * 2 == S, "split");
        const unsigned mask = lane_mask<G>();
        auto sync = [&]() {
            if constexpr (M > 32) __syncthreads();
            else __syncwarp(mask);
        };
        if constexpr (M <= 32) __syncwarp(mask);
        if (g < M) {
#pragma unroll
            for (int m = 0; m < R; ++m) buf[pos(g + M * m)] = x[m];
        }
        sync();
        if (M <= 32 || g < LN) {
            cpx<T> c[CH];
#pragma unroll
            for (int i = 0; i < CH; ++i) {
                const int q = g * CH + i;
                c[i] = buf[pos(q)];
                if (i > 0 || g > 0) c[i] = c[i] + buf[pos(S - q)];   // q = 0: P_0 = V_0 (U_0 = 0)
                if (i > 0) c[i] = c[i - 1] + c[i];
            }
            cpx<T> inc = c[CH - 1];
#pragma unroll
            for (int off = 1; off < LN; off <<= 1) {
                const cpx<T> o = mk<T>(__shfl_up_sync(mask, inc.x, off, LN), __shfl_up_sync(mask, inc.y, off, LN));
                if (g >= off) inc = inc + o;
            }
            cpx<T> ex = mk<T>(__shfl_up_sync(mask, inc.x, 1, LN), __shfl_up_sync(mask, inc.y, 1, LN));
            if (g == 0) ex = mk<T>(0, 0);
            // the sum's other end is known too, V_{S/2-1} = -P_{S/2}: what it misses is spread linearly over the sum,
            // which takes the rounding errors of a random walk to those of a bridge (a third of the variance)
            const cpx<T> end = mk<T>(__shfl_sync(mask, inc.x, LN - 1, LN), __shfl_sync(mask, inc.y, LN - 1, LN));
            const cpx<T> miss = scale(end + buf[pos(S / 2)], (T)(-2.0 / S));
            ex = ex + scale(miss, (T)(g * CH + 1));
#pragma unroll
            for (int i = 0; i < CH; ++i) buf[pos(g * CH + i)] = ex + (c[i] + scale(miss, (T)i));
        }
        sync();
        if (g < M) {
#pragma unroll
            for (int m = 0; m < R; ++m) {
                const int q = g + M * m;
                const cpx<T> v = m < H ? buf[pos(q)] : neg(buf[pos(S - 1 - q)]);   // V_{S-1-q} = -V_q
                x[m] = g < M / 2 ? x[m] - v : v;
            }
            if (g == 0) {   // w_m = U_q at q = M/2 + M m
#pragma unroll
                for (int m = H; m < R; ++m) {
                    const int q = M / 2 + M * m;
                    x[m] = buf[pos(q)] + buf[pos(S - 1 - q)];
                }
            }
        }
    }

    // S <- K_T S on the register values (kf: two rows of G entries per pair of values)
    static __device__ __forceinline__ void kinetic(cpx<T> *x, const D *kf, int g)
    {
#pragma unroll
        for (int pr = 0; pr < NS * H; ++pr) {
            const int e0 = pr / H * R + pr % H, e1 = pr / H * R + R - 1 - pr % H;
            x[e0] = cmul(x[e0], PR::ldd(kf + (2 * pr) * G + g));
            x[e1] = cmul(x[e1], PR::ldd(kf + (2 * pr + 1) * G + g));
        }
    }
};

// ------------------------------------------------------------------------------------------------
// pointwise work.  The step's factor and norm act on the registers (factor_regs), the first and last half-steps
// of a trajectory too.  Everything rarer -- jumps, caps, summary rows, rows beyond the static table, phases beyond
// 1e5, temperatures that change too much within a step, the FP64 KSU factor and the read-out -- works on a copy of
// the registers in shared memory, element e of thread g at e G + g, in loops over e: a thread only touches its own
// elements, and the step's code stays short.
// Values carry the odd extension's sign (fused_plan.h).
// ------------------------------------------------------------------------------------------------
template <typename T, int N, int V> struct Pointwise {
    using P = FusedPlan<T, N, V>;
    using PR = Prec<T>;
    using C = typename Prec<T>::C;
    using SC = typename Prec<T>::S;
    static constexpr int G = P::G, E = P::E, R = P::R, H = P::H, M = P::M, S = P::S, NS = P::NS;
    static constexpr bool RUN = sizeof(T) == 8 && H > 2;   // recurrence along a slot (factor_regs)
    static constexpr bool ADJ = sizeof(T) == 4;   // static rows: the two entries of a pair adjacent

    static __device__ __forceinline__ int jof(int g, int e) { return plan_j(g, e, R, M, G); }
    static __device__ __forceinline__ bool odd_half(int e) { return e % R >= H; }   // the register holds -u_j
    static __device__ __forceinline__ int stat_idx(int g, int e)
    {
        const int m = e % R, h = m >= H, pr = e / R * H + (h ? R - 1 - m : m);
        return ADJ ? 2 * (pr * G + g) + h : (2 * pr + h) * G + g;
    }
    static __device__ __forceinline__ SC stat(const Tables<T> &tb, const SC *tab, int c, int l, int g, int e, bool full)
    {
        if (l < LTAB) return PR::ld_s(&tab[((size_t)c * LTAB + l) * N + stat_idx(g, e)]);
        const int j = jof(g, e);
        if (j == 0) return PR::make_s(0.0, 0.0);
        return static_far<T>(tb.coul[c], tb.M, tb.dt, l, j * tb.dr, full ? 2.0 : 1.0);
    }

    static __device__ __forceinline__ void to_smem(const cpx<T> *x, cpx<T> *buf, int g)
    {
#pragma unroll
        for (int e = 0; e < E; ++e) buf[e * G + g] = x[e];
    }
    static __device__ __forceinline__ void to_regs(cpx<T> *x, const cpx<T> *buf, int g)
    {
#pragma unroll
        for (int e = 0; e < E; ++e) x[e] = buf[e * G + g];
    }

    // The dynamic factor exp(a) exp(i pi y) is close to 1 and changes little from step to step; FP32 applies it
    // as w + w f1 with f1 its deviation from 1, evaluated so that the rounding is relative to f1, not to 1 (a
    // rounding of a value next to 1 would repeat identically every step and add up).  In FP64 a rounding next to 1 does
    // not matter: factor() shares this form, factor_regs multiplies by the factor itself.
    static __device__ __forceinline__ cpx<T> apply(cpx<T> w, T f1r, T f1i)
    {
        if constexpr (sizeof(T) == 4) return mk(fmaf(w.x, f1r, fmaf(-w.y, f1i, w.x)), fmaf(w.y, f1r, fmaf(w.x, f1i, w.y)));
        else return mk(w.x + (w.x * f1r - w.y * f1i), w.y + (w.x * f1i + w.y * f1r));
    }

    // FP64: exp(z j^2), z = A + i Bpi, and the norm weight exp((A + D) j^2) along j = j0 + S m by recurrence,
    // e_{m+1} = e_m h_m, h_{m+1} = h_m q, q = exp(2 z S^2): 10 operations a point and four short series a slot
    // instead of exp and sincospi at every point (60 of the 145 FP64 instructions per point and step at
    // N = 4096, where the FP64 pipe was 86% busy), at a relative error of at most ~m^2/2 roundings (m < R/2).
    struct Run {
        cpx<T> e, h;
        T w, hw;
        template <bool PHASE> __device__ __forceinline__ void start(T A, T B, T D, T j0)
        {
            const T a = j0 * j0, b = (T)S * ((T)2 * j0 + (T)S);
            e = Dyn<double>::template cexp<PHASE>(A * a, B * a, &w);
            h = Dyn<double>::template cexp<PHASE>(A * b, B * b, &hw);
            w *= Dyn<double>::near1(D * a);
            hw *= Dyn<double>::near1(D * b);
        }
        template <bool PHASE> __device__ __forceinline__ void step(cpx<T> qe, T qw)
        {
            if (PHASE) {
                e = e * h;
                h = h * qe;
            } else {
                e.x *= h.x;
                h.x *= qe.x;
            }
            w *= hw;
            hw *= qw;
        }
    };

    // The step's factor on the registers: x <- stat2 dyn_a dyn_b x, accumulating sum exp(2 er_a r^2) |x_old|^2
    // (the end-of-step norm / dr).  dyn = exp((er + i ei) r^2), er and ei multiplied by T^3; A = (er_a + er_b)
    // dr^2, B = (ei_a + ei_b) dr^2 / pi, D = (er_a - er_b) dr^2, rounded once per step and multiplied with the
    // exact j^2 (N <= 4096; rounded once above), so no rounding that repeats identically every step enters.
    // exp(2 er_a r^2) = mag exp((er_a - er_b) r^2), the second factor by its series in z = D j^2 = delta a, with a the
    // exponent of mag and delta = D / A the relative change of the temperature's factor over one step (1.6e-4 for a
    // Bjorken medium at 0.6 fm/c and dt = 0.001): FP32 keeps the first order, FP64 the third.  What the series leave
    // out of mag exp(z) is at most 0.27 delta^2 and 0.2 delta^4 at any a <= 0; the caller keeps |delta| below
    // series_delta, where that is 1e-6 (the FP32 state is some 1e-6 off) and 3e-12, and takes factor() beyond.
    // The first half-step of a trajectory and the last of its last step are the same with the half-step rows and
    // only one half-step's coefficients (last: the sum is |x_new|^2).
    // PHASE = false: gamma_hat = 0, B = 0 exactly, the phase series is skipped (its value would be 0).
    static constexpr T series_delta = (T)(1.0 / 512);
    template <bool PHASE>
    static __device__ __forceinline__ void factor_regs(cpx<T> *x, const SC *row, int g, T A, T B, T D, bool last,
                                                       SqAcc<T> &acc, SqAcc<T> &acc2)
    {
        const T Bpi = (T)3.14159265358979323846 * B;
        const T qlim = fmax(-2 * A, fabs(Bpi));   // a >= -1/2 and |t| <= 1 where qlim j^2 <= 1
        cpx<T> qe;
        T qw;
        if constexpr (RUN) {
            const T s2 = (T)2 * S * S;
            qe = Dyn<double>::template cexp<PHASE>(A * s2, Bpi * s2, &qw);
            qw *= Dyn<double>::near1(D * s2);
        }
#pragma unroll
        for (int t = 0; t < NS; ++t) {
            int lo, hi;
            slot_points(g + t * G, R, M, lo, hi);
            Run ul, uh;
            if constexpr (RUN) {
                ul.template start<PHASE>(A, Bpi, D, (T)lo);
                uh.template start<PHASE>(A, Bpi, D, (T)hi);
            }
#pragma unroll
            for (int m = 0; m < H; ++m) {
                cpx<T> &x0 = x[t * R + m], &x1 = x[t * R + R - 1 - m];
                const int pr = t * H + m;
                if constexpr (sizeof(T) == 4) {
                    // the series of the pair (m, R-1-m) in packed FP32x2 instructions
                    const float4 st = __ldg(reinterpret_cast<const float4 *>(row) + pr * G + g);
                    const float2 j = make_float2((float)(lo + S * m), (float)(hi + S * m));
                    const float2 j2 = __fmul2_rn(j, j);
                    const float2 a2 = __fmul2_rn(make_float2(A, A), j2);
                    float2 fr, fi = make_float2(0.f, 0.f), em;
                    const float2 t2 = __fmul2_rn(make_float2(Bpi, Bpi), j2);
                    // every j of row m is below S (m + 1): one uniform test says that all arguments of the row are
                    // in the series' range
                    const bool near = qlim * ((float)(S * (m + 1)) * (float)(S * (m + 1))) <= 1.0f;
                    if (PHASE) {
                        if (near) Dyn<float>::f1t2(a2, t2, &fr, &fi, &em);
                        else Dyn<float>::far2(a2, t2, &fr, &fi, &em);
                    } else {
                        if (near) em = Dyn<float>::em1_2(a2);
                        else Dyn<float>::far2(a2, t2, &fr, &fi, &em);
                        fr = em;
                    }
                    const float2 mag = __fadd2_rn(make_float2(1.f, 1.f), em);
                    float2 z = __fmul2_rn(make_float2(D, D), j2);
                    z = make_float2(last ? em.x : z.x, last ? em.y : z.y);   // (last: |x_new|^2 = mag^2 |x_old|^2)
                    const float2 wt = __ffma2_rn(mag, z, mag);
                    acc.add_w(x0, wt.x);
                    acc2.add_w(x1, wt.y);
                    const cpx<T> w0 = PR::mul_s(x0, mk(st.x, st.y)), w1 = PR::mul_s(x1, mk(st.z, st.w));
                    x0 = PHASE ? apply(w0, fr.x, fi.x) : mk(fmaf(w0.x, fr.x, w0.x), fmaf(w0.y, fr.x, w0.y));
                    x1 = PHASE ? apply(w1, fr.y, fi.y) : mk(fmaf(w1.x, fr.y, w1.x), fmaf(w1.y, fr.y, w1.y));
                } else {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        cpx<T> &xe = h ? x1 : x0;
                        Run &u = h ? uh : ul;
                        if constexpr (!RUN) {
                            const T j2 = (T)((h ? hi : lo) + S * m) * (T)((h ? hi : lo) + S * m);
                            u.e = Dyn<double>::template cexp<PHASE>(A * j2, Bpi * j2, &u.w);
                            u.w *= Dyn<double>::near1(D * j2);
                        }
                        const cpx<T> w = PR::mul_s(xe, PR::ld_s(row + (2 * pr + h) * G + g));
                        const cpx<T> xn = PHASE ? w * u.e : scale(w, u.e.x);
                        (h ? acc2 : acc).add_w(mk(last ? xn.x : xe.x, last ? xn.y : xe.y), last ? (T)1 : u.w);
                        xe = xn;
                        if (RUN && m + 1 < H) u.template step<PHASE>(qe, qw);
                    }
                }
            }
        }
    }

    // The same in loops over the copy in shared memory, for every mode:
    // mode 0: x <- stat1 dyn_b x (the first half-step of a trajectory)
    // mode 1: x <- stat2 dyn_a dyn_b x; returns sum exp(W j^2) |x_old|^2, W = 2 er_a dr^2 (end-of-step norm / dr)
    // mode 2: x <- stat1 dyn_a x; returns sum |x_new|^2
    static __device__ __noinline__ typename NormSum<T>::type factor(cpx<T> *buf, const Tables<T> &tb, int g, int c, int l,
                                                                    int mode, T A, T B, T W, double *red)
    {
        SqAcc<T> acc;
        const SC *tab = (mode == 1) ? tb.statV2 : tb.statV;
#pragma unroll 4
        for (int e = 0; e < E; ++e) {
            const T fj = (T)jof(g, e);
            T f1r, f1i, em1;
            if constexpr (sizeof(T) == 4) {
                const T j2 = fj * fj;
                Dyn<T>::f1t(A * j2, ((T)3.14159265358979323846 * B) * j2, &f1r, &f1i, &em1);
            } else {
                Dyn<T>::f1((A * fj) * fj, (B * fj) * fj, &f1r, &f1i, &em1);
            }
            cpx<T> v = buf[e * G + g];
            if (mode == 1) acc.add_w(v, k_exp((W * fj) * fj));
            v = apply(PR::mul_s(v, stat(tb, tab, c, l, g, e, mode == 1)), f1r, f1i);
            if (mode == 2) acc.add_w(v, (T)1);
            buf[e * G + g] = v;
        }
        if (mode == 0) return {};
        return slot_norm_sum<T, G>(acc, red);
    }

    // The KSU counterpart of factor (same modes, same w + w f1 form): the dynamic exponent of the
    // half-step at temperature T is (V_I - i (V_R + a/r)) dt/2 at each point, evaluated per point;
    // ka, kb are the per-step scalars of T_n (the closing half-step) and T_{n+1} (the opening one).
    static __device__ typename NormSum<T>::type factor_ksu(cpx<T> *buf, const Tables<T> &tb, int g, int l, int mode,
                                                           const KsuT<T> &ka, const KsuT<T> &kb, double *red)
    {
        SqAcc<T> acc;
        const SC *tab = (mode == 1) ? tb.statV2 : tb.statV;
        const T hdt = (T)0.5 * tb.ksu_dt;
#pragma unroll 2
        for (int e = 0; e < E; ++e) {
            const int j = jof(g, e);
            const T fj = (T)j;
            T A = (T)0, t = (T)0, z = (T)0;
            if (j > 0) {
                T vda = (T)0, via = (T)0, vdb = (T)0, vib = (T)0;
                if (mode != 0) ksu_point<T>(tb, ka, fj, vda, via);
                if (mode != 2) ksu_point<T>(tb, kb, fj, vdb, vib);
                A = (via + vib) * hdt;
                t = -(vda + vdb) * hdt;
                z = (via - vib) * hdt;   // |K_V(n)|^2 = exp(A + z)
            }
            T f1r, f1i, em1;
            if constexpr (sizeof(T) == 4) Dyn<T>::f1t(A, t, &f1r, &f1i, &em1);
            else Dyn<T>::f1(A, t * (T)0.318309886183790671537767526745, &f1r, &f1i, &em1);
            const T mag = (T)1 + em1;
            cpx<T> v = buf[e * G + g];
            if (mode == 1) acc.add_w(v, mag * exp(z));
            const cpx<T> w = PR::mul_s(v, stat(tb, tab, 0, l, g, e, mode == 1));
            v = mk(w.x + (w.x * f1r - w.y * f1i), w.y + (w.x * f1i + w.y * f1r));
            if (mode == 2) acc.add_w(v, (T)1);
            buf[e * G + g] = v;
        }
        if (mode == 0) return {};
        return slot_norm_sum<T, G>(acc, red);
    }

    // A jump after the factor of mode 1 (more steps follow) or mode 2 (after the last step).
    // Returns sum r^2 |end-of-step state|^2 (/ dr); with mode 1 the end-of-step state is
    // exp(-er_b r^2) times the stored one.  With mode 1 it also turns the start half-step already
    // applied from (c, l) into (c2, l2): x <- conj(stat1(c,l)) stat1(c2,l2) exp(d_er r^2 + i d_ei r^2) x.
    // The coefficients come times dr^2 (the phase also / pi) and multiply j^2: w2 = -2 er_b dr^2,
    // A = d_er dr^2, B = d_ei dr^2 / pi.  A one-off factor, so working precision suffices.
    static __device__ double jump_turn(cpx<T> *buf, const Tables<T> &tb, int g, int c, int l, int c2, int l2,
                                       bool after_last, T w2, T A, T B, double *red)
    {
        const T dr2 = (T)(tb.dr * tb.dr);
        SqAcc<T> acc;
#pragma unroll 1
        for (int e = 0; e < E; ++e) {
            const T fj = (T)jof(g, e), j2 = fj * fj;
            cpx<T> v = buf[e * G + g];
            if (after_last) {
                acc.add_w(v, dr2 * j2);
            } else {
                acc.add_w(v, dr2 * j2 * k_exp(w2 * j2));
                v = PR::mul_s(PR::mul_s(v, PR::conj_s(stat(tb, tb.statV, c, l, g, e, false))),
                              stat(tb, tb.statV, c2, l2, g, e, false));
                T sn, cs;
                k_sincospi(B * j2, &sn, &cs);
                const T m = k_exp(A * j2);
                v = v * mk(m * cs, m * sn);
                buf[e * G + g] = v;
            }
        }
        return slot_norm<T, G>(acc, red);
    }

    // Per-step summary row of the end-of-step state e = stat1 exp(A j^2 + i pi B j^2) x, x the state
    // before the closing half-step (A = erj K3, B = eij T3 of the step): norm, <r>, overlaps, FP64
    // accumulation; thread 0 writes the row.  One pass for the norm and <r> and one per basis state
    // of the same l, so that few values stay live.  Only in the traced kernels (V = 4, 6).
    static __device__ __forceinline__ cpx<double> end_value(const cpx<T> *buf, const Tables<T> &tb, int c, int l, int g,
                                                            int e, T A, T B)
    {
        const T fj = (T)jof(g, e);
        T f1r, f1i, em1;
        Dyn<T>::f1((A * fj) * fj, (B * fj) * fj, &f1r, &f1i, &em1);
        const cpx<T> w = PR::mul_s(buf[e * G + g], stat(tb, tb.statV, c, l, g, e, false));
        return mk((double)(w.x + (w.x * f1r - w.y * f1i)), (double)(w.y + (w.x * f1i + w.y * f1r)));
    }

    static __device__ void trace_row(const cpx<T> *buf, const Tables<T> &tb, int g, int c, int l, T A, T B,
                                     double *red, qtraj_trace_rec *out, int step)
    {
        double n2 = 0.0, rr = 0.0;
#pragma unroll 1
        for (int e = 0; e < E; ++e) {
            const cpx<double> v = end_value(buf, tb, c, l, g, e, A, B);
            const double m2 = v.x * v.x + v.y * v.y;
            n2 += m2;
            rr += (double)jof(g, e) * tb.dr * m2;
        }
        n2 = slot_sum<G>(n2, red);
        rr = slot_sum<G>(rr, red);
        const double dr = tb.dr;
        if (g == 0) {
            out->step = step;
            out->color = c;
            out->l = l;
            out->flags = 0;
            out->norm2 = n2 * dr;
            out->r_ratio = (rr / n2) / tb.r1s;
        }
#pragma unroll 1
        for (int s = 0; s < NBASIS; ++s) {
            const int bl = s == 2 || s == 4 ? 1 : (s == 5 ? 2 : 0);
            double vr = 0.0, vi = 0.0;
            if (c == 0 && bl == l) {
#pragma unroll 1
                for (int e = 0; e < E; ++e) {
                    const cpx<double> v = end_value(buf, tb, c, l, g, e, A, B);
                    const double phi = tb.eig[(size_t)s * N + jof(g, e)], ph = odd_half(e) ? -phi : phi;
                    vr += ph * v.x;
                    vi += ph * v.y;
                }
                vr = slot_sum<G>(vr, red);
                vi = slot_sum<G>(vi, red);
            }
            if (g == 0) out->ov2[s] = (vr * vr + vi * vi) * dr / n2;
        }
    }

    // Undoes the start half-step applied by a mode-1 factor, x <- conj(stat1(c,l)) exp(A j^2 + i pi B j^2) x
    // with A = -er_b dr^2 and B = -ei_b dr^2 / pi: the end-of-step state of a trajectory that stops
    // at a jump cap.
    static __device__ void undo_start(cpx<T> *buf, const Tables<T> &tb, int g, int c, int l, T A, T B)
    {
#pragma unroll 1
        for (int e = 0; e < E; ++e) {
            const T fj = (T)jof(g, e), j2 = fj * fj;
            T sn, cs;
            k_sincospi(B * j2, &sn, &cs);
            const T m = k_exp(A * j2);
            buf[e * G + g] = PR::mul_s(buf[e * G + g], PR::conj_s(stat(tb, tb.statV, c, l, g, e, false))) * mk(m * cs, m * sn);
        }
    }

    // fin <- the sums of the read-out (norm^2 / dr, overlaps / dr with the nb basis states of l) of an FP32 state in FP64
    static __device__ __noinline__ void read_out64(const cpx<T> *buf, const Tables<T> &tb, int g, int nb, int l, double *red,
                                                   double *fin)
    {
        double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        const double *phi = tb.eig + (size_t)(l == 0 ? 0 : l == 1 ? 2 : 5) * N;   // 1S 2S . 3S, 1P . 2P, 1D
#pragma unroll 1
        for (int e = 0; e < E; ++e) {
            const int j = jof(g, e);
            const double sg = odd_half(e) ? -1.0 : 1.0, x = sg * (double)buf[e * G + g].x, y = sg * (double)buf[e * G + g].y;
            v[0] = fma(x, x, fma(y, y, v[0]));
#pragma unroll
            for (int i = 0; i < 3; ++i)
                if (i < nb) {
                    const double f = phi[(size_t)(l == 1 ? 2 * i : i == 2 ? 3 : i) * N + j];
                    v[1 + 2 * i] = fma(f, x, v[1 + 2 * i]);
                    v[2 + 2 * i] = fma(f, y, v[2 + 2 * i]);
                }
        }
        slot_sums8<G>(v, red, fin);
    }

    // x <- x * r_j * f
    static __device__ void scale_r(cpx<T> *buf, const Tables<T> &tb, int g, double f)
    {
        const T s = (T)(tb.dr * f);
#pragma unroll 1
        for (int e = 0; e < E; ++e) buf[e * G + g] = scale(buf[e * G + g], (T)jof(g, e) * s);
    }
};

// the ready flag of a group's no-jump record, with acquire semantics: the record written before the
// flag was released is visible after it
__device__ __forceinline__ int group_ready(const int *p)
{
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// a record written by another CTA of this launch, read past L1
__device__ __forceinline__ qtraj_obs load_obs_cg(const qtraj_obs *p)
{
    static_assert(sizeof(qtraj_obs) % 8 == 0, "qtraj_obs is a whole number of 8-byte words");
    qtraj_obs o;
    const unsigned long long *src = reinterpret_cast<const unsigned long long *>(p);
    unsigned long long *dst = reinterpret_cast<unsigned long long *>(&o);
#pragma unroll
    for (int i = 0; i < (int)(sizeof(qtraj_obs) / 8); ++i) dst[i] = __ldcg(src + i);
    return o;
}

// One thread per CTA takes work items from the counter: a group's no-jump run (item < n_groups) or a
// trajectory; r0 < p_NoJump (once the group's record is ready, or from a previous launch's records)
// and r0 > r_max are resolved here without evolving.
template <typename T>
__device__ int fetch_trajectory(const Tables<T> &tb, const LaunchArgs &a)
{
    for (;;) {
        const int w = atomicAdd(a.counter, 1);
        if (w >= a.n_groups + a.n_traj) return -1;
        if (a.nojump || w < a.n_groups) return w;
        const int t = w - a.n_groups;
        const TrajDev d = a.trajs[t];
        const Draws dr0 = draws(d.seed, 0u);
        int flags = 0;
        bool have = false;   // p_NoJump known (its group's record is published), or no shortcut at all
        if (tb.use_rmin) {
            qtraj_obs gj;
            if (a.gready) {
                if (group_ready(a.gready + d.group)) {
                    gj = load_obs_cg(a.gobs + d.group);
                    have = true;
                }
            } else if (a.group) {
                gj = a.group[d.group];
                have = true;
            }
            if (have) {
                if (fabs(dr0.r - gj.norm2) < border_eps<T>()) flags |= QTRAJ_F_BORDERLINE;
                if (dr0.r < gj.norm2) {
                    qtraj_obs o = gj;
                    o.r0 = dr0.r;
                    o.n_steps_exec = 0;
                    o.flags = flags | QTRAJ_F_NOJUMP_SHORTCUT;
                    a.obs[t] = o;
                    continue;
                }
            }
        }
        // r0 > r_max is resolved only once r0 < p_NoJump is excluded; otherwise the kernel evolves it
        if (tb.potential == 0 && dr0.r > tb.r_max && (have || !tb.use_rmin)) {
            qtraj_obs o;
            for (int s = 0; s < NBASIS; ++s) { o.surv[s] = 0; o.ov_re[s] = 0; o.ov_im[s] = 0; }
            o.norm2 = 1.0;
            o.r0 = dr0.r;
            o.l = tb.spec_l[d.spec];
            o.color = tb.spec_color[d.spec];
            o.n_jumps = 0;
            o.n_steps_exec = 0;
            o.flags = flags | QTRAJ_F_RMAX;
            o.first_jump_step = -1;
            o.last_jump_step = -1;
            o.jump_digest = DIGEST_BASIS;
            a.obs[t] = o;
            continue;
        }
        return w;
    }
}

constexpr int fused_red = 8;   // sums reduced at once (slot_sums8)

// Occupancy target of a kernel variant: variant 0 asks for 512 resident threads per SM in FP32
// (<= 128 registers); variant 1 asks for 640 (N = 2048: 5 CTAs of 128 threads, <= 102 registers, at the price of
// spills; at N = 4096 640 threads hold the same two CTAs of 256), variants 2 and 3 (radix 8) for 768 and 1024.  FP64 holds twice the state and takes what the compiler needs.
template <typename T, int N, int V> struct FusedBounds {
    static constexpr int G = FusedPlan<T, N, V>::G;
    static constexpr int THREADS = V == 1 ? 640 : V == 2 || V == 6 ? 768 : V == 3 ? 1024 : 512;
    static constexpr int MB = THREADS / G > 32 ? 32 : (THREADS / G > 0 ? THREADS / G : 1);
    static constexpr int MIN_BLOCKS = sizeof(T) == 4 ? MB : 1;
};

template <typename T, int N, int V>
__global__ void __launch_bounds__(FusedPlan<T, N, V>::G, (FusedBounds<T, N, V>::MIN_BLOCKS)) fused_kernel(Tables<T> tb, LaunchArgs a)
{
    using P = FusedPlan<T, N, V>;
    using K = Sine<T, N, V>;
    using PW = Pointwise<T, N, V>;
    using NS2 = typename NormSum<T>::type;
    constexpr int G = P::G, E = P::E, NS = P::NS, RED = fused_red;
    constexpr bool KSU = V == 5;                  // the isotropic KSU potential: H_eff only, no jumps
    constexpr bool TRACED = V == 4 || V == 6;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cpx<T> *buf = reinterpret_cast<cpx<T> *>(smem_raw);
    double *red = reinterpret_cast<double *>(buf + P::BUF);         // reductions of the rare paths
    NS2 *redh = reinterpret_cast<NS2 *>(red + RED * (G / 32 + 1) + 8);  // the step's norm
    __shared__ int s_traj;

    const int g = threadIdx.x;
    const double dr = tb.dr;
    int pb[NS], pm[NS];
#pragma unroll
    for (int t = 0; t < NS; ++t) {
        int lo, hi;
        slot_points(g + t * G, P::R, P::M, lo, hi);
        pb[t] = K::pos(lo);
        pm[t] = K::pos(P::S - lo);   // (slot 0 does not use them)
    }
    cpx<T> x[P::XN];

    for (;;) {
        if (g == 0) s_traj = fetch_trajectory(tb, a);
        __syncthreads();
        const int wk = s_traj;
        __syncthreads();
        if (wk < 0) break;
        const bool grp = wk < a.n_groups;     // a group's no-jump run of this launch
        const int t = grp ? wk : wk - a.n_groups;
        const bool nojump = a.nojump || grp || KSU;

        const TrajDev *dp = grp ? a.gtrajs + t : a.trajs + t;
        const int spec = dp->spec, ns = dp->n_steps;
        const MediumDev *mp = tb.media + dp->medium;
        int l = tb.spec_l[spec], c = tb.spec_color[spec];
        {
            const double *ic = tb.ic + (size_t)spec * N * (tb.ic_cplx ? 2 : 1);
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int j = PW::jof(g, e);
                const T re = tb.ic_cplx ? (T)ic[2 * j] : (T)ic[j], im = tb.ic_cplx ? (T)ic[2 * j + 1] : (T)0;
                x[e] = PW::odd_half(e) ? mk(-re, -im) : mk(re, im);
            }
        }
        uint32_t kdraw = 0;
        Threshold<T> thr;
        // r0 > r_max reaches here only when its group's no-jump record was not yet published: the paper
        // resolves r0 < p_NoJump by the shortcut first and r0 > r_max only otherwise.  The trajectory
        // is evolved: if its norm never falls to r0 it is the no-jump run (= the shortcut's record); the
        // first trigger shows r0 >= p_NoJump (the norm only decreases), and it ends as r_max does.
        bool rmax_pending = false;
        {
            const double r = nojump ? -1.0 : draws(dp->seed, 0u).r;   // (no draw is used without jumps)
            thr.set(r, dr);
            rmax_pending = !nojump && r > tb.r_max;
        }
        int nj = 0, flags = 0, fj = -1, lj = -1, ended = 0, executed = 0;
        uint32_t digest = DIGEST_BASIS;
        bool rmax_hit = false;
        const bool traced = TRACED && !grp && a.trace_every > 0 && t < a.trace_n;
        int nrec = 0;
        int seg = 0;
        // T(tau_n)^3: Bjorken, or the table at tau_n = tau_1 + n dtau (out of line: rare, and inline it
        // would hold registers in the step loop)
        auto T3_of = [&](int n) -> T {
            const T tau = (T)mp->tau0 + (T)n * (T)mp->dtau;
            return mp->kind == 1 ? table_T3_far<T>(tb.prof + 2 * (size_t)mp->tab_off, mp->tab_len, tau, &seg)
                                 : (T)mp->A / tau;
        };
        T T3b = (T)0, K3b = (T)0;   // K3: kappa_hat(T) T^3 when kappa_hat follows a lattice fit
        KsuT<T> kb{};
        bool in_smem = false;   // the state is in the shared-memory copy (else in the registers)

        // step -1 is the first half-step alone, so that the factor's code is there once
        for (int n = ns > 0 ? -1 : 0; n < ns; ++n) {
            const T T3a = T3b, K3a = K3b;
            const bool start = n < 0, last = n + 1 == ns;
            T3b = T3_of(n + 1);
            K3b = kappa_T3<T>(mp->kfit, T3b);
            in_smem = false;
            if (!start) {
#pragma unroll 1
                for (int h = 0; h < 2; ++h) {
                    K::first(x, buf, tb.TA, tb.TH, g, pb, pm);
                    traj_sync<G>();
                    K::mid(x, buf, tb.TM, tb.TI, tb.TS, g);
                    traj_sync<G>();
                    K::last(x, buf, tb.TM, g);
                    if (h == 0) {
                        K::kinetic(x, tb.KF, g);
                        traj_sync<G>();
                    }
                }
            }
            executed = n + 1;
            const T erj = (T)mp->erj[c], eij = (T)mp->eij[c];
            if constexpr (TRACED) {   // per-step summary rows
                if (!start && traced && ((n + 1) % a.trace_every == 0 || last) && nrec < a.trace_cap) {
                    traj_sync<G>();
                    PW::to_smem(x, buf, g);
                    PW::trace_row(buf, tb, g, c, l, erj * K3a, eij * T3a, red,
                                  a.trace + (size_t)t * a.trace_cap + nrec, n + 1);
                    ++nrec;
                }
            }
            const T Tsum = last ? T3a : T3a + T3b, Ksum = last ? K3a : K3a + K3b;   // (step -1: T3a = K3a = 0)
            const T cA = erj * Ksum, cB = eij * Tsum, cD = start || last ? (T)0 : erj * (K3a - K3b);
            const int mode = start ? 0 : last ? 2 : 1;
            NS2 n2s;   // norm^2 / dr
            // (phases beyond 1e5: far2's reduction would lose them; a temperature that changes by more within a step than
            // the norm's weight allows: steep tabulated media, or dt above 0.01 in a Bjorken medium at 0.6 fm/c.  The latter test
            // costs a trajectory of one warp 55 ns a step, N = 256 through 96 steps 329 -> 338 us; larger grids < 0.5%)
            if (KSU || l >= LTAB || !(fabs(cB) * (T)N * (T)N < (T)3e4) || fabs(cD) > PW::series_delta * fabs(cA)) {
                traj_sync<G>();   // all have read the transform's output
                PW::to_smem(x, buf, g);
                in_smem = true;
                if constexpr (KSU) {
                    const KsuT<T> ka = kb;
                    kb = ksu_at<T>(tb, T3b);
                    n2s = PW::factor_ksu(buf, tb, g, l, mode, ka, kb, red);
                } else {
                    n2s = PW::factor(buf, tb, g, c, l, mode, cA, cB, 2 * erj * K3a, red);
                }
            } else {
                SqAcc<T> acc, acc2;
                const typename Prec<T>::S *row = (mode == 1 ? tb.statV2 : tb.statV) + ((size_t)c * LTAB + l) * N;
                if (cB == (T)0) PW::template factor_regs<false>(x, row, g, cA, cB, cD, last, acc, acc2);
                else PW::template factor_regs<true>(x, row, g, cA, cB, cD, last, acc, acc2);
                acc.merge(acc2);
                n2s = step_norm<T, G>(acc, redh);   // synchronises: all have read the transform's output
            }
            if (start) {
                if (in_smem) {
                    PW::to_regs(x, buf, g);
                    traj_sync<G>();   // the copies are read before the first pass writes its sequences
                }
                continue;
            }
            bool stop = false;
            if (!thr.finite(n2s)) {
                flags |= QTRAJ_F_NONFINITE;
                ended = 1;
                if (g == 0) atomicOr(a.status, 1);
                stop = true;
            } else if (!nojump) {
                if (thr.near(n2s, border_eps<T>())) flags |= QTRAJ_F_BORDERLINE;
                if (thr.reached(n2s)) {
                    if (!in_smem) PW::to_smem(x, buf, g);
                    in_smem = true;
                    const Draws dw = draws(dp->seed, kdraw);
                    // a trajectory stopped by a cap keeps its end-of-step state
                    const bool cap_j = tb.max_jumps >= 0 && nj >= tb.max_jumps;
                    const int l_new = (dw.ul < (double)l / (2.0 * l + 1.0)) ? l - 1 : l + 1;
                    const int c_new = (c == 1 && dw.uc < tb.p_os) ? 0 : 1;
                    const bool cap_l = !cap_j && tb.l_cap >= 0 && l_new > tb.l_cap;
                    if (rmax_pending) {
                        rmax_hit = true;
                        ended = 1;
                        stop = true;
                    } else if (cap_j || cap_l) {
                        if (!last) PW::undo_start(buf, tb, g, c, l, -(T)mp->erj[c] * K3b, -(T)mp->eij[c] * T3b);
                        ended = 1;
                        if (cap_j) {
                            flags |= QTRAJ_F_MAXJUMPS;
                        } else {
                            flags |= QTRAJ_F_LCAP;
                            if (fj < 0) fj = n;
                            l = l_new; c = c_new; ++nj;
                            lj = n;
                            digest = digest_jump(digest, n, l, c);
                        }
                        stop = true;
                    } else {
                        if (fj < 0) fj = n;
                        // r times the end-of-step state, renormalised; the start half-step already applied
                        // is turned into the new colour's and l's
                        const double dr2 = tb.dr * tb.dr, T3d = (double)T3b, K3d = (double)K3b;
                        const T w2 = last ? (T)0 : (T)(-2.0 * mp->er[c] * K3d * dr2);
                        const T dA = last ? (T)0 : (T)((mp->er[c_new] - mp->er[c]) * K3d * dr2);
                        const T dB = last ? (T)0 : (T)((mp->ei[c_new] - mp->ei[c]) * T3d * dr2 * 0.31830988618379067154);
                        const double s = PW::jump_turn(buf, tb, g, c, l, c_new, l_new, last, w2, dA, dB, red) * dr;
                        PW::scale_r(buf, tb, g, 1.0 / sqrt(s));
                        l = l_new; c = c_new; ++nj;
                        lj = n;
                        digest = digest_jump(digest, n, l, c);
                        ++kdraw;
                        thr.set(draws(dp->seed, kdraw).r, dr);
                    }
                }
            }
            if (stop) break;
            if (in_smem && !last) {
                PW::to_regs(x, buf, g);
                traj_sync<G>();
            }
        }

        // (all have read the transform's output: step_norm, or the sync before the copy)
        if (!in_smem) PW::to_smem(x, buf, g);

        // the norm and the overlaps of the state's l in one pass over the shared-memory copy, in FP64 or (FP32) in
        // error-free parts: the sums ran on the FP64 pipe before, 160 of its instructions a warp of 16 values a thread
        double *fin = red + 8 * (G / 32 + 1);   // norm^2 / dr, then (re, im) / dr of each overlap
        const int nb = ended || c != 0 || l > 2 ? 0 : 3 - l;            // basis states of this l: 1S 2S 3S, 1P 2P, 1D
        auto state_of = [&](int i) { return l == 0 ? (i == 2 ? 3 : i) : l == 1 ? 2 + 2 * i : 5; };
        auto observe = [&](auto n) {
            constexpr int NB = decltype(n)::value;
            using Dot = typename std::conditional<sizeof(T) == 4, Dot2, Dot1>::type;
            using RL = typename Prec<T>::Rl;
            Dot norm, dot[NB > 0 ? NB : 1];
            const RL *phi[NB > 0 ? NB : 1];
#pragma unroll
            for (int i = 0; i < NB; ++i) phi[i] = tb.eigo + (size_t)state_of(i) * N + g;
#pragma unroll 4
            for (int e = 0; e < E; ++e) {
                const cpx<T> u = buf[e * G + g];
                if constexpr (sizeof(T) == 4) norm.add(make_float2(u.x, u.y), make_float2(u.x, u.y));
                else norm.sq(u);
#pragma unroll
                for (int i = 0; i < NB; ++i) {
                    if constexpr (sizeof(T) == 4) dot[i].add(Prec<T>::ldr(phi[i] + e * G), make_float2(u.x, u.y));
                    else dot[i].add(__ldg(phi[i] + e * G), u);
                }
            }
            double v[8] = {norm.x() + norm.y(), 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
            for (int i = 0; i < NB; ++i) {
                v[1 + 2 * i] = dot[i].x();
                v[2 + 2 * i] = dot[i].y();
            }
            slot_sums8<G>(v, red, fin);
        };
        if (nb == 0) observe(std::integral_constant<int, 0>{});
        else if (nb == 3) observe(std::integral_constant<int, 3>{});
        else if (nb == 2) observe(std::integral_constant<int, 2>{});
        else observe(std::integral_constant<int, 1>{});
        if constexpr (sizeof(T) == 4) {
            traj_sync<G>();
            if (ns == 0 || !dot2_holds(fin[0])) PW::read_out64(buf, tb, g, nb, l, red, fin);
        }
        if (a.states && !grp) {
            double *st = a.states + (size_t)t * N * 2;
#pragma unroll 4
            for (int e = 0; e < E; ++e) {
                const cpx<T> v = buf[e * G + g];
                const int j = PW::jof(g, e);
                const double sg = PW::odd_half(e) ? -1.0 : 1.0;
                st[2 * j] = sg * (double)v.x;
                st[2 * j + 1] = sg * (double)v.y;
            }
        }
        // the record: a lane of the first warp per basis state, the rest by thread 0
        if (g < 32) {
            qtraj_obs *o = grp ? a.gobs + t : a.obs + t;
            const double n2 = fin[0] * dr;
            for (int s = g; s < NBASIS; s += G < 32 ? G : 32) {
                const int sl = s == 2 || s == 4 ? 1 : s == 5 ? 2 : 0, i = s < 3 ? (s == 2 ? 0 : s) : s == 3 ? 2 : s == 4 ? 1 : 0;
                double re = 0.0, im = 0.0, sv = 0.0;
                if (nb > 0 && sl == l && !rmax_hit) {
                    re = fin[1 + 2 * i] * dr;
                    im = fin[2 + 2 * i] * dr;
                    // with jumps the estimator takes the normalised state; without (KSU) the norm lost to V_I is
                    // the dissociation, and the overlap is taken unnormalised
                    sv = (re * re + im * im) / (KSU ? 1.0 : n2);
                    if (!tb.ov0_zero[spec * NBASIS + s]) {
                        const double a0 = tb.ov0[(spec * NBASIS + s) * 2], b0 = tb.ov0[(spec * NBASIS + s) * 2 + 1];
                        sv /= a0 * a0 + b0 * b0;
                    }
                }
                o->surv[s] = sv;
                o->ov_re[s] = re;
                o->ov_im[s] = im;
            }
            if (grp) __threadfence();         // the record before the flag that publishes it
            __syncwarp(lane_mask<G>());
            if (g == 0) {
                o->norm2 = rmax_hit ? 1.0 : n2;
                o->r0 = nojump ? 0.0 : draws(dp->seed, 0u).r;
                // (rmax_hit: the r_max record, with the steps that found r0 >= p_NoJump)
                o->l = rmax_hit ? tb.spec_l[spec] : l;
                o->color = rmax_hit ? tb.spec_color[spec] : c;
                o->n_jumps = nj;
                o->n_steps_exec = executed;
                o->flags = rmax_hit ? flags | QTRAJ_F_RMAX : flags;
                o->first_jump_step = fj;
                o->last_jump_step = lj;
                o->jump_digest = digest;
                if (grp) {
                    __threadfence();
                    atomicExch(a.gready + t, 1);
                }
                if (traced) a.trace_cnt[t] = nrec;
            }
        }
        __syncthreads();
    }
}

// shared-memory bytes of one CTA
template <typename T, int N, int V> constexpr int fused_smem_bytes()
{
    using P = FusedPlan<T, N, V>;
    return P::BUF * (int)sizeof(cpx<T>) + (P::G / 32 + 1) * (fused_red + 1) * 8 + 64;
}

// Launches a trajectory kernel as one persistent wave (SMs x resident CTAs, at most max_ctas when
// max_ctas > 0, at most one CTA per trajectory) after setting its shared-memory size; fills info
// (query_only: launches nothing).
template <typename T>
cudaError_t launch_wave(void (*k)(Tables<T>, LaunchArgs), int G, int R, int smem, const Tables<T> &tb, const LaunchArgs &a,
                        int sm_count, int max_ctas, cudaStream_t s, FusedInfo *info, bool query_only)
{
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    int occ = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, G, smem);
    if (e != cudaSuccess) return e;
    if (occ < 1) return cudaErrorInvalidConfiguration;
    if (info) {
        cudaFuncAttributes fa;
        e = cudaFuncGetAttributes(&fa, k);
        if (e != cudaSuccess) return e;
        info->G = G;
        info->R = R;
        info->smem = smem;
        info->ctas_per_sm = occ;
        info->regs = fa.numRegs;
    }
    const long work = (long)a.n_traj + a.n_groups;
    if (query_only || work <= 0) return cudaSuccess;
    long grid = (long)sm_count * occ;
    if (max_ctas > 0 && grid > max_ctas) grid = max_ctas;
    if (grid > work) grid = work;
    k<<<(int)grid, G, smem, s>>>(tb, a);
    return cudaGetLastError();
}

// Every instantiation unit dispatches its grid sizes to this helper.
template <typename T, int N, int V>
cudaError_t fused_go(const Tables<T> &tb, const LaunchArgs &a, int sm_count, int max_ctas, cudaStream_t s,
                     FusedInfo *info, bool query_only)
{
    using P = FusedPlan<T, N, V>;
    return launch_wave(fused_kernel<T, N, V>, P::G, P::R, fused_smem_bytes<T, N, V>(), tb, a, sm_count, max_ctas, s, info,
                       query_only);
}

} // namespace qt
