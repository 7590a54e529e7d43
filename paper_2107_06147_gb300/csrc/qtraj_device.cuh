// qtraj_device.cuh -- device-side building blocks shared by the fused and the plain forms:
// complex arithmetic, Philox4x32-10, small in-register DFTs, and the device records.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "qtraj.h"

namespace qt {

constexpr int NBASIS = QTRAJ_NBASIS;
constexpr int LTAB = 256;            // l rows per colour of the static space-kernel tables
constexpr double BORDER_EPS = 1e-12; // |norm^2 - r| below this flags a borderline comparison (FP64)
// The FP32 forms flag at the error of their norm instead: the state is carried in FP32, and its
// norm after thousands of steps is good to ~1e-6 (the paired FP32/FP64 study: 3e-4 of the jumps
// moved by a step, at ~3e-3 mean norm change per step between jumps), so a threshold closer to the
// norm than that may be crossed a step earlier or later than in exact arithmetic.
constexpr double BORDER_EPS_F32 = 1e-6;
template <typename T> __host__ __device__ constexpr double border_eps()
{
    return sizeof(T) == 4 ? BORDER_EPS_F32 : BORDER_EPS;
}

// ------------------------------------------------------------------------------------------------
// complex numbers
// ------------------------------------------------------------------------------------------------
template <typename T> struct alignas(2 * sizeof(T)) cpx { T x, y; };

template <typename T> __host__ __device__ __forceinline__ cpx<T> mk(T a, T b) { return {a, b}; }
template <typename T> __device__ __forceinline__ cpx<T> operator+(cpx<T> a, cpx<T> b) { return {a.x + b.x, a.y + b.y}; }
template <typename T> __device__ __forceinline__ cpx<T> operator-(cpx<T> a, cpx<T> b) { return {a.x - b.x, a.y - b.y}; }
template <typename T> __device__ __forceinline__ cpx<T> operator*(cpx<T> a, cpx<T> b)
{
    return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
template <typename T> __device__ __forceinline__ cpx<T> scale(cpx<T> a, T s) { return {a.x * s, a.y * s}; }
template <typename T> __device__ __forceinline__ cpx<T> mul_i(cpx<T> a) { return {-a.y, a.x}; }   // i*a
template <typename T> __device__ __forceinline__ cpx<T> mul_mi(cpx<T> a) { return {a.y, -a.x}; }  // -i*a
// FP32: complex add, subtract and real scale as packed FP32x2 instructions (sm_100 and later): both
// components in one instruction, each with the same IEEE rounding as the scalar form (a - b is
// fma(-1, b, a), exact in the product), so results are bit-identical and the issue slots halve
template <> __device__ __forceinline__ cpx<float> operator+(cpx<float> a, cpx<float> b)
{
    const float2 r = __fadd2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y));
    return {r.x, r.y};
}
template <> __device__ __forceinline__ cpx<float> operator-(cpx<float> a, cpx<float> b)
{
    const float2 r = __ffma2_rn(make_float2(-1.f, -1.f), make_float2(b.x, b.y), make_float2(a.x, a.y));
    return {r.x, r.y};
}
template <> __device__ __forceinline__ cpx<float> scale(cpx<float> a, float s)
{
    const float2 r = __fmul2_rn(make_float2(a.x, a.y), make_float2(s, s));
    return {r.x, r.y};
}
// read-only-cache loads of complex values
__device__ __forceinline__ cpx<float> ldg(const cpx<float> *p)
{
    const float2 v = __ldg(reinterpret_cast<const float2 *>(p));
    return {v.x, v.y};
}
__device__ __forceinline__ cpx<double> ldg(const cpx<double> *p)
{
    const double2 v = __ldg(reinterpret_cast<const double2 *>(p));
    return {v.x, v.y};
}
// ------------------------------------------------------------------------------------------------
// constant multipliers.  The rounding of a constant is the same in every step and accumulates coherently over
// 10^4 steps, while the rounding of data is random and grows only as a square root.  So the FP32 constants of the
// transforms and the kinetic factors carry more than 24 bits: complex ones as directions (Prec<float>::D, 2^-35), real
// ones, and all of the FP32 KSU kernel's, as unevaluated sums hi + lo of two floats (2^-48).  The static potential
// rows are single floats.  In FP64 a constant is one double.
// ------------------------------------------------------------------------------------------------
template <typename T> struct Prec;
template <> struct Prec<double> {
    using C = cpx<double>; // complex constant
    using Rl = double;     // real constant
    static __host__ C make(double re, double im) { return {re, im}; }
    static __host__ __device__ Rl make_r(double v) { return v; }
    static __device__ __forceinline__ cpx<double> mul(cpx<double> x, C w) { return x * w; }
    static __device__ __forceinline__ C conj(C w) { return {w.x, -w.y}; }
    using D = C;           // (FP32: a direction, below)
    static __device__ __forceinline__ D ncj(D w) { return {-w.x, w.y}; }
    static __device__ __forceinline__ cpx<double> muld(cpx<double> x, D w) { return x * w; }
    static __device__ __forceinline__ D ldd(const D *p) { return ldg(p); }
    static __device__ __forceinline__ cpx<double> mulr(cpx<double> x, Rl s) { return scale(x, s); }
    static __device__ __forceinline__ C ld(const C *p) { return ldg(p); }
    static __device__ __forceinline__ Rl re(C w) { return w.x; }
    static __device__ __forceinline__ Rl im(C w) { return w.y; }
    // static potential factors (tables of exp(-i V_static dt/2), exp(-i V_static dt)): one double each
    using S = cpx<double>;
    static __host__ __device__ S make_s(double re, double im) { return {re, im}; }
    static __device__ __forceinline__ S ld_s(const S *p) { return ldg(p); }
    static __device__ __forceinline__ cpx<double> mul_s(cpx<double> x, S w) { return x * w; }
    static __device__ __forceinline__ S conj_s(S w) { return {w.x, -w.y}; }
};
template <> struct Prec<float> {
    struct alignas(16) C { float rh, ih, rl, il; };
    struct alignas(8) Rl { float h, l; };
    static __host__ C make(double re, double im)
    {
        const float rh = (float)re, ih = (float)im;
        return {rh, ih, (float)(re - (double)rh), (float)(im - (double)ih)};
    }
    static __host__ __device__ Rl make_r(double v)
    {
        const float h = (float)v;
        return {h, (float)(v - (double)h)};
    }
    static __device__ __forceinline__ cpx<float> mul(cpx<float> x, C w)
    {
        const float lr = fmaf(x.x, w.rl, -x.y * w.il), li = fmaf(x.x, w.il, x.y * w.rl);
        return {fmaf(x.x, w.rh, fmaf(-x.y, w.ih, lr)), fmaf(x.x, w.ih, fmaf(x.y, w.rh, li))};
    }
    static __device__ __forceinline__ C conj(C w) { return {w.rh, -w.ih, w.rl, -w.il}; }
    // A complex constant as a direction, (r + i im)(1 + d): of the float pairs whose larger component is within 4096
    // steps of the constant's, the one whose direction is nearest (about 2^-37 off), and the real factor that is
    // left, |d| < 2^-11, itself good to 2^-35.  A product takes 6 operations instead of the 8 of hi + lo parts, which
    // were a quarter of a step's; the 2^-35 repeat in every step, far below the 2^-24 roundings of the data that
    // average out over 10^4 steps.
    struct alignas(16) D { float r, im, d, pad; };
    static __device__ __forceinline__ D ncj(D w) { return {-w.r, w.im, w.d, 0.f}; }
    static __device__ __forceinline__ cpx<float> muld(cpx<float> x, D w)
    {
        const float a = fmaf(x.x, w.r, -x.y * w.im), b = fmaf(x.x, w.im, x.y * w.r);
        return {fmaf(a, w.d, a), fmaf(b, w.d, b)};
    }
    static __device__ __forceinline__ D ldd(const D *p)
    {
        const float4 v = __ldg(reinterpret_cast<const float4 *>(p));
        return {v.x, v.y, v.z, 0.f};
    }
    static __device__ __forceinline__ cpx<float> mulr(cpx<float> x, Rl s)
    {
        return {fmaf(x.x, s.h, x.x * s.l), fmaf(x.y, s.h, x.y * s.l)};
    }
    static __device__ __forceinline__ C ld(const C *p)
    {
        const float4 v = __ldg(reinterpret_cast<const float4 *>(p));
        return {v.x, v.y, v.z, v.w};
    }
    static __device__ __forceinline__ Rl ldr(const Rl *p)
    {
        const float2 v = __ldg(reinterpret_cast<const float2 *>(p));
        return {v.x, v.y};
    }
    static __device__ __forceinline__ Rl re(C w) { return {w.rh, w.rl}; }
    static __device__ __forceinline__ Rl im(C w) { return {w.ih, w.il}; }
    // The static potential factors are the one family of constants kept without low parts: the
    // paired FP32/FP64 study measured no loss from rounding them (ensemble errors 1.6e-6 / 1.1e-5 at
    // N = 4096 / 8192 against 2.6e-6 / 4.2e-6 with hi+lo; median norm error 6.7e-7 against 5.3e-7),
    // while their table is the one a trajectory reads per (colour, l) row -- half the bytes.
    using S = cpx<float>;
    static __host__ __device__ S make_s(double re, double im) { return {(float)re, (float)im}; }
    static __device__ __forceinline__ S ld_s(const S *p) { return ldg(p); }
    static __device__ __forceinline__ cpx<float> mul_s(cpx<float> x, S w)
    {
        return {fmaf(x.x, w.x, -x.y * w.y), fmaf(x.x, w.y, x.y * w.x)};
    }
    static __device__ __forceinline__ S conj_s(S w) { return {w.x, -w.y}; }
};

// a * (rh + i ih) with the constant's low parts (rl, il) in FP32; plain product in FP64
template <typename T> __device__ __forceinline__ cpx<T> mulk(cpx<T> a, double re, double im)
{
    if constexpr (sizeof(T) == 4) {
        const Prec<float>::C w{(float)re, (float)im, (float)(re - (double)(float)re), (float)(im - (double)(float)im)};
        return Prec<float>::mul(a, w);
    } else {
        return a * mk<T>(re, im);
    }
}
template <typename T> __device__ __forceinline__ T mulkr(T v, double c)
{
    if constexpr (sizeof(T) == 4) return fmaf(v, (float)c, v * (float)(c - (double)(float)c));
    else return v * c;
}

template <typename T> __device__ __forceinline__ double abs2d(cpx<T> a)
{
    return (double)a.x * (double)a.x + (double)a.y * (double)a.y;
}

// ------------------------------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): counter (k,0,0,0), key = 64-bit seed.
// Waiting period k of a trajectory uses the four words of counter k: the threshold r from words
// 0 and 1 (53 bits), the angular-momentum draw u_l from word 2 and the colour draw u_c from word 3.
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ void philox10(uint32_t &c0, uint32_t &c1, uint32_t &c2, uint32_t &c3, uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int i = 0; i < 10; ++i) {
        if (i) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
        const uint32_t lo0 = 0xD2511F53u * c0, hi0 = __umulhi(0xD2511F53u, c0);
        const uint32_t lo1 = 0xCD9E8D57u * c2, hi1 = __umulhi(0xCD9E8D57u, c2);
        const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
        c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
    }
}

struct Draws { double r, ul, uc; };

// the jump digest of a record: 32-bit FNV-1a over the little-endian bytes of (step, new l, new colour)
// of every jump in order
constexpr uint32_t DIGEST_BASIS = 2166136261u;
__host__ __device__ __forceinline__ uint32_t digest_word(uint32_t h, uint32_t w)
{
#pragma unroll
    for (int b = 0; b < 4; ++b) h = (h ^ ((w >> (8 * b)) & 255u)) * 16777619u;
    return h;
}
__host__ __device__ __forceinline__ uint32_t digest_jump(uint32_t h, int step, int l, int c)
{
    return digest_word(digest_word(digest_word(h, (uint32_t)step), (uint32_t)l), (uint32_t)c);
}

__device__ __forceinline__ Draws draws(unsigned long long seed, uint32_t k)
{
    uint32_t c0 = k, c1 = 0, c2 = 0, c3 = 0;
    philox10(c0, c1, c2, c3, (uint32_t)seed, (uint32_t)(seed >> 32));
    const unsigned long long w = ((unsigned long long)c1 << 32) | c0;
    Draws d;
    d.r = ((double)(w >> 11) + 0.5) * 0x1.0p-53;
    d.ul = ((double)c2 + 0.5) * 0x1.0p-32;
    d.uc = ((double)c3 + 0.5) * 0x1.0p-32;
    return d;
}

// ------------------------------------------------------------------------------------------------
// in-register DFTs of size 2, 4, 8, 16: X_k = sum_n x_n exp(-2 pi i n k / R), natural order in/out
// ------------------------------------------------------------------------------------------------
// x * exp(-2 pi i j/16) for a compile-time j (after unrolling the switch folds away); the constants
// cos(pi/8), sin(pi/8), sqrt(1/2) enter with their FP32 low parts in the FP32 form
template <typename T> __device__ __forceinline__ cpx<T> tw16(cpx<T> a, int j)
{
    constexpr double c1 = 0.92387953251128675613, s1 = 0.38268343236508977173, h = 0.70710678118654752440;
    switch (j & 15) {
    case 0: return a;
    case 1: return mulk<T>(a, c1, -s1);
    case 2: return mk(mulkr<T>(a.x + a.y, h), mulkr<T>(a.y - a.x, h));
    case 3: return mulk<T>(a, s1, -c1);
    case 4: return mul_mi(a);
    case 5: return mulk<T>(a, -s1, -c1);
    case 6: return mk(mulkr<T>(a.y - a.x, h), mulkr<T>(-a.x - a.y, h));
    case 7: return mulk<T>(a, -c1, -s1);
    case 8: return mk(-a.x, -a.y);
    case 9: return mulk<T>(a, -c1, s1);
    case 10: return mk(mulkr<T>(-a.x - a.y, h), mulkr<T>(a.x - a.y, h));
    case 11: return mulk<T>(a, -s1, c1);
    case 12: return mul_i(a);
    case 13: return mulk<T>(a, s1, c1);
    case 14: return mk(mulkr<T>(a.x - a.y, h), mulkr<T>(a.x + a.y, h));
    default: return mulk<T>(a, c1, s1);
    }
}

// x * exp(-2 pi i j/32) for a compile-time j, the constants as directions (Prec<float>::D) in FP32
template <typename T> __device__ __forceinline__ cpx<T> tw32(cpx<T> a, int j)
{
    // cos and sin of pi/16, pi/8 and 3 pi/16, and the nearest directions: (c, s)(1 + d) within 7e-12
    constexpr double cs[3][2] = {{0.98078528040323044913, 0.19509032201612826785},
                                 {0.92387953251128675613, 0.38268343236508977173},
                                 {0.83146961230254523708, 0.55557023301960222474}};
    constexpr float fd[3][3] = {{0.980871439f, 0.19510746f, -8.78388091e-05f},
                                {0.923697054f, 0.382607847f, 0.000197551912f},
                                {0.831550539f, 0.555624306f, -9.73196875e-05f}};
    j &= 31;
    if (j % 4 == 0) return tw16<T>(a, j / 2);   // multiples of pi/4
    // reduce to the first octant: angle j pi/16 = quadrant + (o or 8 - o)
    const int o = j % 8, k = (o < 4 ? o : 8 - o) - 1;
    const bool sw = o > 4;
    const int quad = j / 8;   // (-i)^quad (c - i s)
    auto rot = [&](auto c, auto s, auto &re, auto &im) {
        re = quad == 0 ? c : quad == 1 ? -s : quad == 2 ? -c : s;
        im = quad == 0 ? -s : quad == 1 ? -c : quad == 2 ? s : c;
    };
    if constexpr (sizeof(T) == 4) {
        float re, im;
        rot(sw ? fd[k][1] : fd[k][0], sw ? fd[k][0] : fd[k][1], re, im);
        return Prec<float>::muld(a, Prec<float>::D{re, im, fd[k][2], 0.f});
    } else {
        double re, im;
        rot(sw ? cs[k][1] : cs[k][0], sw ? cs[k][0] : cs[k][1], re, im);
        return a * mk<T>(re, im);
    }
}

template <typename T> __device__ __forceinline__ void dft2(cpx<T> &a, cpx<T> &b)
{
    const cpx<T> t = a;
    a = t + b;
    b = t - b;
}

template <typename T> __device__ __forceinline__ void dft4(cpx<T> &x0, cpx<T> &x1, cpx<T> &x2, cpx<T> &x3)
{
    const cpx<T> a = x0 + x2, b = x0 - x2, c = x1 + x3, d = mul_mi(x1 - x3);
    x0 = a + c;
    x2 = a - c;
    x1 = b + d;
    x3 = b - d;
}

// DFT of R = R1*R2 points held at x[base + stride*n]: inner DFTs of size R1 over n1 (n = R2 n1 + n2),
// twiddles W_R^{n2 k1}, outer DFTs of size R2 over n2; output index k = k1 + R1 k2.
template <typename T, int R> struct DFT;

template <typename T> struct DFT<T, 1> {
    template <int S> __device__ __forceinline__ static void run(cpx<T> *) {}
};
template <typename T> struct DFT<T, 2> {
    template <int S> __device__ __forceinline__ static void run(cpx<T> *x) { dft2(x[0], x[S]); }
};
template <typename T> struct DFT<T, 4> {
    template <int S> __device__ __forceinline__ static void run(cpx<T> *x) { dft4(x[0], x[S], x[2 * S], x[3 * S]); }
};
template <typename T> struct DFT<T, 8> {
    template <int S> __device__ __forceinline__ static void run(cpx<T> *x)
    {
        // n = 2 n1 + n2: two DFT4 over n1, twiddle W8^{n2 k1}, four DFT2 over n2
        cpx<T> y[8];
#pragma unroll
        for (int n2 = 0; n2 < 2; ++n2) {
            cpx<T> a = x[(0 + n2) * S], b = x[(2 + n2) * S], c = x[(4 + n2) * S], d = x[(6 + n2) * S];
            dft4(a, b, c, d);
            y[n2 * 4 + 0] = a;
            y[n2 * 4 + 1] = tw16(b, 2 * n2 * 1);
            y[n2 * 4 + 2] = tw16(c, 2 * n2 * 2);
            y[n2 * 4 + 3] = tw16(d, 2 * n2 * 3);
        }
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            cpx<T> a = y[k1], b = y[4 + k1];
            dft2(a, b);
            x[(k1)*S] = a;
            x[(k1 + 4) * S] = b;
        }
    }
};
template <typename T> struct DFT<T, 16> {
    template <int S> __device__ __forceinline__ static void run(cpx<T> *x)
    {
        // n = 4 n1 + n2: four DFT4 over n1, twiddle W16^{n2 k1}, four DFT4 over n2
        cpx<T> y[16];
#pragma unroll
        for (int n2 = 0; n2 < 4; ++n2) {
            cpx<T> a = x[(0 + n2) * S], b = x[(4 + n2) * S], c = x[(8 + n2) * S], d = x[(12 + n2) * S];
            dft4(a, b, c, d);
            y[n2 * 4 + 0] = a;
            y[n2 * 4 + 1] = tw16(b, n2 * 1);
            y[n2 * 4 + 2] = tw16(c, n2 * 2);
            y[n2 * 4 + 3] = tw16(d, n2 * 3);
        }
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            cpx<T> a = y[k1], b = y[4 + k1], c = y[8 + k1], d = y[12 + k1];
            dft4(a, b, c, d);
            x[(k1)*S] = a;
            x[(k1 + 4) * S] = b;
            x[(k1 + 8) * S] = c;
            x[(k1 + 12) * S] = d;
        }
    }
};

// ------------------------------------------------------------------------------------------------
// device records
// ------------------------------------------------------------------------------------------------
struct MediumDev {
    double A;       // T0^3 tau0, so T(tau_n)^3 = A / (tau0 + n dtau)  (kind 0)
    double tau0;    // fm/c: tau of step 0 (kind 1: the table's first tau)
    double dtau;    // dt * hbar c, fm/c per step
    double er[2];   // -kappa_c dt/2 per colour: the real exponent of the space kernel is er*T^3*r^2
    double ei[2];   // -gamma_c dt/2 per colour: the phase of the space kernel is ei*T^3*r^2
    double erj[2];  // er * dr^2: the real exponent is erj * T^3 * j^2 on grid point j
    double eij[2];  // ei * dr^2 / pi: the phase is pi * eij * T^3 * j^2
    int kfit;       // 0: constant kappa_hat, folded into er/erj; 1, 2, 3: er/erj are per unit kappa_hat
                    // and T^3 in the real exponent becomes kappa_hat(T) T^3 from lattice fit kfit
    int kind;       // 0 Bjorken; 1 tabulated: points [tab_off, tab_off + tab_len) of the profile store
    int tab_off, tab_len;
};

// T^3 at tau of a tabulated medium, p = its (tau, T) pairs: linear in T between the neighbouring
// points, the first/last T outside.  seg is the caller's segment index (p[seg].tau <= tau), moved
// forward only, so a trajectory walks its table once.
template <typename T> __device__ __forceinline__ T table_T3(const double *p, int len, T tau, int &seg)
{
    while (seg + 2 < len && tau >= (T)p[2 * (seg + 1)]) ++seg;
    const T t0 = (T)p[2 * seg], t1 = (T)p[2 * seg + 2], T0 = (T)p[2 * seg + 1], T1 = (T)p[2 * seg + 3];
    T f = (tau - t0) / (t1 - t0);
    f = f < (T)0 ? (T)0 : (f > (T)1 ? (T)1 : f);
    const T Tt = T0 + f * (T1 - T0);
    return Tt * Tt * Tt;
}

// the same from scratch (binary search), for kernels that do not carry a segment index
__device__ __forceinline__ double table_T3_at(const double *p, int len, double tau)
{
    int lo = 0, hi = len - 1;   // find the last point with tau_i <= tau, at most len - 2
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (p[2 * mid] <= tau) lo = mid;
        else hi = mid;
    }
    int seg = lo;
    return table_T3<double>(p, len, tau, seg);
}

// kappa_hat(T) T^3 given T^3: kfit 0 returns T^3 (kappa_hat is folded into the exponent's
// coefficient); kfit 1, 2, 3 multiply by the central, lower or upper lattice fit of the Munich
// potential (App. E), kappa_hat = 1 / (a x^{3/2} + b x + c x^{1/2} + d) with x = T / T_c,
// T_c = 0.155 GeV, evaluated in the working precision once per step.
template <typename T> __device__ __forceinline__ T kappa_T3(int kfit, T T3)
{
    if (kfit == 0) return T3;
    const T a = kfit == 1 ? (T)0.00397 : kfit == 2 ? (T)0.00712 : (T)0.00272;
    const T b = kfit == 1 ? (T)-0.08341 : kfit == 2 ? (T)-0.14262 : (T)-0.05854;
    const T c = kfit == 1 ? (T)0.98031 : kfit == 2 ? (T)1.55601 : (T)0.71513;
    const T d = kfit == 1 ? (T)-0.51889 : kfit == 2 ? (T)-0.80712 : (T)-0.38197;
    const T s = sqrt(cbrt(T3) * (T)(1.0 / 0.155));
    return T3 / (((a * s + b) * s + c) * s + d);
}

struct TrajDev {
    unsigned long long seed;
    int spec, medium, n_steps, group;
};

static_assert(sizeof(qtraj_obs) == 192, "qtraj_obs layout");
static_assert(sizeof(qtraj_trace_rec) == 80, "qtraj_trace_rec layout");

// Read-only context tables (device pointers) and scalars.
template <typename T> struct Tables {
    using C = typename Prec<T>::C;
    // FP32 KSU kernel, natural order
    const C *W;                        // N twiddles exp(-2 pi i t / N)
    const C *WL;                       // last-pass twiddles W^(m g), [R][N/(2R)] (ksu32_wl_radix)
    const C *KT;                       // N kinetic factors exp(-i T_kin(p_k) dt) * 2/N, k = 0..N-1
    const typename Prec<T>::Rl *sinpre; // N values sin(pi j / N)
    // both forms, in the order of the kernels' threads (fused_plan.h)
    using D = typename Prec<T>::D;
    const D *KF;                       // N kinetic factors exp(-i T_kin(p_k) dt) * (-1/(2N))
    const D *TA;                       // first-pass twiddles W_2N^(b k): [R/2 - 1][N/R], k = 1 .. R/2 - 1
    const C *TH;                       // the same for k = R/2: [N/R]
    const D *TM;                       // W_S^(b1 q1): [b1][q1] applied by the last pass, else [q1][b1]
    const C *TS;                       // [R/2] (1/(2 sin(pi k/R)), cot(pi k/R)/2): the sequences' positions 0, S/2
    const D *TI;                       // between two middle passes: W_M^(m2 k1), [k1][m2]
    const typename Prec<T>::S *statV;  // [2][LTAB][N] exp(-i (V_coul + l(l+1)/(M r^2)) dt/2)
    const typename Prec<T>::S *statV2; // [2][LTAB][N] the same over a full step, exp(-i (...) dt)
                                       // (both in natural order for the FP32 KSU kernel)
    const double *eig;     // [NBASIS][N] Coulomb basis, discretely normalised
    const typename Prec<T>::Rl *eigo;   // the same in the order e G + g of the fused kernel's values, with their signs
    const double *ic;      // initial states, discretely normalised: [n_spec][N] real, or
                           // [n_spec][N][2] (re, im) when ic_cplx (after a vacuum evolution)
    const double *ov0;     // [n_spec][NBASIS][2] initial overlaps
    const int *ov0_zero;   // [n_spec][NBASIS] structural zero of the initial overlap
    const int *spec_l;     // [n_spec]
    const int *spec_color; // [n_spec]
    const MediumDev *media;
    double dr, dt, M, p_os;
    double coul[2];        // coefficient of 1/r of the colour's Coulomb potential
    int max_jumps, l_cap, use_rmin;
    double r_max;
    int ic_cplx;
    const double *prof;    // profile store: (tau, T) pairs of the tabulated media
    double r1s;            // <1S|r|1S> on the grid (discrete), the unit of the summary's R
    // the isotropic KSU potential (potential = 1; App. E), see qtraj_params.potential:
    int potential;
    const T *phi_tab;      // (phi, h phi') at a = KSU_PHI_A0 + i h, i < KSU_PHI_NODES (h = 1/KSU_PHI_PER)
    const T *phi_ser;      // [KSU_PHI_SER][2]: the small-argument series of phi, coefficients of y^k
                           // (y = a^2) of the ln a part and of the rest (k = 1 ..)
    T ksu_a_dr;            // a / dr: the Coulomb part a/r = ksu_a_dr / j
    T ksu_sig_dr;          // sigma dr: the linear part sigma r = ksu_sig_dr j
    T ksu_two_sigma;       // 2 sigma
    T ksu_cap;             // V_vac(r_SB) = -a/r_SB + sigma r_SB
    T ksu_alpha0, ksu_b0, ksu_mu0sq;   // alpha_s(mu) = alpha0 / (1 + alpha0 b0 ln(mu^2 / mu0^2))
    T ksu_md2;             // F_mD^2 Nc (1 + N_F/6) pi C_F: m_D^2 = ksu_md2 T^2 alpha_s(2 pi T)
    T ksu_cf;              // C_F
    T ksu_dt;              // the step (GeV^-1) in the working precision
};
constexpr double KSU_PHI_A0 = 0.5, KSU_PHI_A1 = 40.0;
constexpr int KSU_PHI_PER = 256;                                   // nodes per unit of a
constexpr int KSU_PHI_NODES = (int)((KSU_PHI_A1 - KSU_PHI_A0) * KSU_PHI_PER) + 1;
constexpr int KSU_PHI_SER = 8;                                     // series terms (a < KSU_PHI_A0)

// per-launch arguments of both forms
struct LaunchArgs {
    const TrajDev *trajs;
    int n_traj;
    qtraj_obs *obs;         // per trajectory (main mode) or per group (no-jump mode)
    const qtraj_obs *group; // no-jump records read by the shortcut (main mode)
    int *counter;           // work counter (fused) -- zeroed before the launch
    int *status;            // bit 0: a non-finite norm was seen
    double *states;         // optional final states [n_traj][N] complex128
    int nojump;             // 1: no-jump mode (trajectory t = group t, never jumps)
    qtraj_trace_rec *trace; // per-step summary rows [trace_n][trace_cap] (traced kernel; off if trace_every 0)
    int *trace_cnt;         // rows written per traced trajectory
    int trace_every, trace_n, trace_cap;
    // fused form, one launch for the rMin shortcut: work items [0, n_groups) are the no-jump runs of
    // the groups (gtrajs -> gobs, then gready[g] = 1), items n_groups + t the trajectories.  A
    // trajectory fetched after its group's flag is set takes the shortcut; one fetched before runs
    // its whole medium, which gives the same record (the shortcut is exact) but counts its steps.
    const TrajDev *gtrajs;
    int n_groups;
    qtraj_obs *gobs;
    int *gready;
};

} // namespace qt
