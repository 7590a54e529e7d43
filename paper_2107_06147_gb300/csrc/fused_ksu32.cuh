// fused_ksu32.cuh -- the FP32 kernel of the isotropic KSU potential (App. E; no jumps): one CTA evolves one
// trajectory, its wave function in shared memory for its whole life, as fused.cuh's kernel does, with the
// sine transform taken through one N-point FFT with sine pre- and post-processing and a compensated prefix
// sum.  fused.cuh's transform is faster and more accurate.  It is not taken here yet because it would move results:
// the KSU survival ratios are referred to the overlaps of the initial state with the Cornell basis, and where one
// of these nearly vanishes the ratio magnifies the two transforms' FP32 difference, to more than 2e-5 of a batch's ratios
// (relative 2-norm) for 25% of Gaussian widths in 0.7 .. 0.9 GeV^-1 on N = 4096, 16 steps, while states and
// overlaps differ by no more than this transform's own error there, 1e-5.
//
// The DST-I of the N-point complex vector f (f_0 = f_N = 0) is computed with one N-point complex FFT:
//   y_j = sin(pi j/N)(f_j + f_{N-j}) + (f_j - f_{N-j})/2,   Y = FFT_N(y),
//   S_{2k}   = (i/2)(Y_k - Y_{N-k}),
//   S_{2k+1} = S_{2k-1} + (Y_k + Y_{N-k})/2,  S_{-1} = -S_1    (a prefix sum over k < N/2).
// In shared memory S is kept as S_{2k} at [k] and S_{2k+1} at [N/2 + k + k/R] (the padded "odd area").
//
// FFT: Stockham autosort with radices R (first pass), MID = N/R^2 in passes of <= 16, R (last).
// Thread g of G = N/(2R) owns butterflies b1 = g, b2 = N/R - g (g = 0: 0 and N/(2R)) of the first
// and last passes, i.e. the indices b + m N/R, m < R.  Those index sets are closed under j -> N - j,
// so the pre- and post-processing, which pair j with N - j, stay inside a thread's registers.
// Shared-memory addresses of the FFT passes are padded by one element every R.
#pragma once
#include "fused.cuh"

namespace qt {

template <int N> struct NftPlan {
    // radix 8 up to N = 2048 (passes 8, 16, 8 at N = 1024 and 8, 16, 2, 8 at 2048: +9% each over
    // radix 16's 16, 4, 16 and 16, 8, 16, whose short middle passes and small CTAs cost more
    // instructions per point), 16 above
    static constexpr int R = ksu32_radix(N);
    static constexpr int G = N / (2 * R);        // threads per trajectory
    static constexpr int NR = N / R;             // stride of a first/last-pass butterfly
    static constexpr int MID = N / (R * R);      // product of the middle radices
    static constexpr int M1 = MID >= 16 ? 16 : MID;
    static constexpr int M2 = MID / M1;          // 1, 2, 4, 8 or 16
    static constexpr int BUF = N + N / R + 8;    // padded FFT extent; also holds the E/odd layout
    // middle-pass twiddle tables in shared memory, row m holding W^(m k) for the k of every thread
    // (tw1: [M1][R] of W_{R M1}; tw2: [M2][R M1] of W_{R M1 M2}), so that a warp reads consecutive
    // entries.  (A flat table W^t read at t = m k with one pad entry every 8 met up to 7-way bank
    // conflicts at odd m -- 44% of the step's shared-memory conflicts at N = 4096.)
    static constexpr int TW1 = R * M1;
    static constexpr int TW2 = M2 > 1 ? R * M1 * M2 : 0;
    static_assert(N == R * M1 * M2 * R, "plan");
    // shared memory without the cached potential: state, twiddles, carries and reductions
    static constexpr int SMEM = BUF * 8 + (TW1 + TW2) * 16 + (G / 32 + 1) * (16 + 64) + 64;
    static constexpr int MIN_BLOCKS = 512 / G > 32 ? 32 : (512 / G > 0 ? 512 / G : 1);   // 512 threads per SM
    // the potential at T_{n+1} is cached where that costs no resident CTA (N <= 2048)
    static constexpr bool CACHE = (SMEM + N * 8) * MIN_BLOCKS <= 220 * 1024;
};


// compensated complex value for the scan's carries between threads.  Chunk totals use cascaded
// summation (the TwoSum error terms are collected separately); carries between threads are
// double-float additions.  The rounding of a chunk total is added to every later odd coefficient
// (a step in k, energy growing with the number of coefficients after it): with plain FP32 chunk
// totals the no-jump FP32 norm drifted by +7e-9 per step at N = 1024 (against < 5e-9 compensated),
// so the 3% they would save at N = 4096 is not taken.
struct Carry {
    DF re{0.f, 0.f}, im{0.f, 0.f};
    __device__ __forceinline__ void add(cpx<float> a)
    {
        const DF r = two_sum(re.hi, a.x), i = two_sum(im.hi, a.y);
        re = DF{r.hi, re.lo + r.lo};
        im = DF{i.hi, im.lo + i.lo};
    }
    __device__ __forceinline__ void add(const Carry &o) { re = df_add(re, o.re); im = df_add(im, o.im); }
    __device__ __forceinline__ cpx<float> plus(cpx<float> a) const   // this + a, one rounding of the sum
    {
        return mk((re.hi + a.x) + re.lo, (im.hi + a.y) + im.lo);
    }
    __device__ __forceinline__ Carry shfl_up(unsigned mask, int off, int w) const
    {
        Carry o;
        o.re = DF{__shfl_up_sync(mask, re.hi, off, w), __shfl_up_sync(mask, re.lo, off, w)};
        o.im = DF{__shfl_up_sync(mask, im.hi, off, w), __shfl_up_sync(mask, im.lo, off, w)};
        return o;
    }
};
template <int N> struct NftSine {
    using T = float;
    using P = NftPlan<N>;
    using PR = Prec<T>;
    using C = typename Prec<T>::C;
    using RL = typename Prec<T>::Rl;
    static constexpr int R = P::R, G = P::G, NR = P::NR, E = 2 * R;
    using DR = DFTI<T, R, true>;
    static __device__ __forceinline__ cpx<T> cmul(cpx<T> x, C w) { return PR::mul(x, w); }

    static __device__ __forceinline__ int pad(int j) { return j + j / R; }
    // E/odd layout of the transform's output (and of the state between transforms): S_{2k} at
    // even_pos(k), S_{2k+1} at odd_pos(k).  (An XOR swizzle of both areas, meant to spread the
    // even/odd lanes of the transform's load over all banks, measured 0.4-4.6% slower.)
    static __device__ __forceinline__ int even_pos(int k) { return k; }
    static __device__ __forceinline__ int odd_pos(int k) { return N / 2 + k + k / R; }
    static __device__ __forceinline__ int b_of(int g, int t) { return t == 0 ? (g == 0 ? 0 : g) : (g == 0 ? NR / 2 : NR - g); }
    // global index of register element e (first/last-pass layout)
    static __device__ __forceinline__ int idx(int g, int e) { return b_of(g, e / R) + (e % R) * NR; }
    // shared-memory position of S_j in the E/odd layout
    static __device__ __forceinline__ int s_pos(int j) { return (j & 1) ? odd_pos(j >> 1) : even_pos(j >> 1); }

    // y_j = s (f_j + f_{N-j}) + (f_j - f_{N-j})/2 for the pair (ea, eb) = (j, N-j)
    static __device__ __forceinline__ void pre_pair(cpx<T> *x, int ea, int eb, RL s)
    {
        const cpx<T> a = x[ea], b = x[eb];
        const cpx<T> sum = PR::mulr(a + b, s), dif = scale(a - b, (T)0.5);
        x[ea] = sum + dif;
        x[eb] = sum - dif;
    }

    static __device__ __forceinline__ void pre(cpx<T> *x, int g, const RL *sinpre)
    {
        if (g != 0) {
#pragma unroll
            for (int m = 0; m < R; ++m) pre_pair(x, m, R + (R - 1 - m), PR::ldr(&sinpre[g + m * NR]));
        } else {
            x[0] = mk<T>(0, 0);                                // j = 0
            x[R / 2] = scale(x[R / 2], (T)2);                  // j = N/2 pairs with itself, sin = 1
#pragma unroll
            for (int m = 1; m < R / 2; ++m) pre_pair(x, m, R - m, PR::ldr(&sinpre[m * NR]));
#pragma unroll
            for (int m = 0; m < R / 2; ++m) pre_pair(x, R + m, R + (R - 1 - m), PR::ldr(&sinpre[NR / 2 + m * NR]));
        }
    }

    // E_k = (i/2)(Y_k - Y_{N-k}) -> [k];  C_k = (Y_k + Y_{N-k})/2 (C_0 halved) -> odd area
    static __device__ __forceinline__ void post_pair(cpx<T> *buf, int k, cpx<T> A, cpx<T> B)
    {
        buf[even_pos(k)] = mul_i(scale(A - B, (T)0.5));
        buf[odd_pos(k)] = scale(A + B, (T)0.5);
    }

    // Y at index b_t + m NR is in register slot t R + operm(m) after the last pass
    static __device__ __forceinline__ cpx<T> Y(const cpx<T> *x, int t, int m) { return x[t * R + DR::operm(m)]; }

    static __device__ __forceinline__ void post(const cpx<T> *x, int g, cpx<T> *buf)
    {
        if (g != 0) {
#pragma unroll
            for (int m = 0; m < R; ++m) {
                if (m < R / 2) post_pair(buf, g + m * NR, Y(x, 0, m), Y(x, 1, R - 1 - m));
                else post_pair(buf, (NR - g) + (R - 1 - m) * NR, Y(x, 1, R - 1 - m), Y(x, 0, m));
            }
        } else {
            buf[even_pos(0)] = mk<T>(0, 0);
            buf[odd_pos(0)] = scale(Y(x, 0, 0), (T)0.5);      // S_1 = C_0 / 2 = Y_0 / 2
#pragma unroll
            for (int m = 1; m < R / 2; ++m) post_pair(buf, m * NR, Y(x, 0, m), Y(x, 0, R - m));
#pragma unroll
            for (int m = 0; m < R / 2; ++m) post_pair(buf, NR / 2 + m * NR, Y(x, 1, m), Y(x, 1, R - 1 - m));
        }
    }

    // inclusive prefix sum of the N/2 odd-area values: thread g owns the chunk k in [gR, gR + R).
    // Chunk totals and the carries between chunks are compensated (a rounding error there would reach
    // every later coefficient); the running sum inside a chunk is plain and only reaches its chunk.
    static __device__ __forceinline__ void scan(cpx<T> *buf, int g, Carry *wtot)
    {
        constexpr int W = G < 32 ? G : 32;
        const unsigned mask = lane_mask<G>();
        cpx<T> v[R];
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = buf[odd_pos(g * R + q)];
        Carry tot;
#pragma unroll
        for (int q = 0; q < R; ++q) tot.add(v[q]);
        const int lane = threadIdx.x & (W - 1);
        Carry inc = tot;
#pragma unroll
        for (int off = 1; off < W; off <<= 1) {
            Carry y = inc.shfl_up(mask, off, W);
            if (lane >= off) inc.add(y);
        }
        Carry excl = inc.shfl_up(mask, 1, W);
        if (lane == 0) excl = Carry();
        if constexpr (G > 32) {
            const int warp = threadIdx.x >> 5;
            if (lane == 31) wtot[warp] = inc;
            __syncthreads();
#pragma unroll 1
            for (int w = 0; w < warp; ++w) excl.add(wtot[w]);
        }
        cpx<T> run = mk<T>(0, 0);
#pragma unroll
        for (int q = 0; q < R; ++q) {
            run = run + v[q];
            buf[odd_pos(g * R + q)] = excl.plus(run);
        }
    }

    // One middle pass (radix RM after PP points): butterfly i reads [i + m N/RM], multiplies by
    // W_{PP RM}^{m k} (k = i mod PP) and writes [(i - k) RM + k + m PP].  A thread's butterflies are
    // g + q G; when PP <= G they share k = g mod PP and so their twiddles, which are loaded once per m
    // (from tw, the table [RM][PP] of W_{PP RM}^{m k}).
    template <int RM, int PP>
    static __device__ __forceinline__ void mid_pass(cpx<T> *x, cpx<T> *buf, const C *tw, int g)
    {
        if constexpr (RM > 1) {
            constexpr int NB = N / RM, PER = E / RM;
            static_assert(PP <= G, "mid-pass twiddle sharing needs PP <= G");
            const int k = g & (PP - 1);
#pragma unroll
            for (int m = 0; m < RM; ++m) {
                C w{};
                if (m) w = tw_at(tw, m * PP + k);
#pragma unroll
                for (int q = 0; q < PER; ++q) {
                    cpx<T> v = buf[pad(g + q * G + m * NB)];
                    if (m) v = cmul(v, w);
                    x[q * RM + m] = v;
                }
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                const int i = g + q * G;
                DFTI<T, RM, true>::run(x + q * RM);
                const int base = (i - k) * RM + k;
#pragma unroll
                for (int m = 0; m < RM; ++m) buf[pad(base + m * PP)] = x[q * RM + DFTI<T, RM, true>::operm(m)];
            }
            __syncthreads();
        }
    }

    static __device__ __forceinline__ C tw_at(const C *tw, int i)
    {
        const float4 v = *reinterpret_cast<const float4 *>(tw + i);
        return C{v.x, v.y, v.z, v.w};
    }

    // S (E/odd layout in buf), optionally times K_T, at the first-pass indices -> DST -> E/odd layout
    static __device__ __forceinline__ void dst(cpx<T> *x, cpx<T> *buf, const Tables<T> &tb, int g, Carry *wtot,
                                               const C *tw1, const C *tw2, bool kinetic)
    {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int j = idx(g, e);
            cpx<T> v = buf[s_pos(j)];
            if (kinetic) v = cmul(v, PR::ld(&tb.KT[j]));
            x[e] = v;
        }
        __syncthreads();
        pre(x, g, tb.sinpre);
        // first pass (radix R, no twiddles): butterfly b -> [b R + k]
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            DR::run(x + t * R);
            const int b = b_of(g, t);
#pragma unroll
            for (int k = 0; k < R; ++k) buf[pad(b * R + k)] = x[t * R + DR::operm(k)];
        }
        __syncthreads();
        mid_pass<P::M1, R>(x, buf, tw1, g);
        mid_pass<P::M2, R * P::M1>(x, buf, tw2, g);
        // last pass (radix R, stride N/R): inputs [b + m NR], twiddle W^(m b).  For the mirror butterfly
        // b2 = NR - g, W^(m b2) = W_R^m conj(W^(m g)): one table load serves both (g = 0 pairs
        // 0 with NR/2, whose twiddles are loaded directly).
#pragma unroll
        for (int m = 0; m < R; ++m) {
            cpx<T> v1 = buf[pad(b_of(g, 0) + m * NR)];
            cpx<T> v2 = buf[pad(b_of(g, 1) + m * NR)];
            if (m) {
                // W^(m g): up to N = 2048 from the compact [m][g] table (a warp reads
                // consecutive entries; measured +3% at N = 1024, +6.5% at 2048), above from the
                // strided W[m g] (the compact table measured 9% slower at N = 4096, 1% at 16384)
                const C w = ksu32_wl_radix(N) ? PR::ld(&tb.WL[m * G + g])
                                      : PR::ld(&tb.W[m * g]);
                v1 = cmul(v1, w);
                if (g != 0) {
                    v2 = tw16<T>(cmul(v2, PR::conj(w)), m * (16 / R));
                } else {
                    v2 = cmul(v2, PR::ld(&tb.W[m * (NR / 2)]));
                }
            }
            x[m] = v1;
            x[R + m] = v2;
        }
        __syncthreads();
#pragma unroll
        for (int t = 0; t < 2; ++t) DR::run(x + t * R);
        post(x, g, buf);
        __syncthreads();
        scan(buf, g, wtot);
        __syncthreads();
    }
};

// ------------------------------------------------------------------------------------------------
// pointwise work on the E/odd layout: thread g visits k = g, g + G, ... < N/2 and the two elements
// S_{2k} (at even_pos(k) = k) and S_{2k+1} (at odd_pos(k))
// ------------------------------------------------------------------------------------------------
template <int N> struct NftPointwise {
    using T = float;
    using K = NftSine<N>;
    using PR = Prec<T>;
    static constexpr int G = K::G;
    using SC = typename Prec<T>::S;
    static __device__ __forceinline__ SC stat(const Tables<T> &tb, const SC *tab, int c, int l, int j, bool full)
    {
        if (l < LTAB) return PR::ld_s(&tab[((size_t)c * LTAB + l) * N + j]);
        if (j == 0) return PR::make_s(0.0, 0.0);
        return static_far<T>(tb.coul[c], tb.M, tb.dt, l, j * tb.dr, full ? 2.0 : 1.0);
    }

    // the read-out's sums in FP64 (Pointwise::read_out64)
    static __device__ __noinline__ void read_out64(const cpx<T> *buf, const Tables<T> &tb, int g, int nb, int l, double *red,
                                                   double *fin)
    {
        double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        const double *phi = tb.eig + (size_t)(l == 0 ? 0 : l == 1 ? 2 : 5) * N;
#pragma unroll 1
        for (int j = 2 * g; j < N; j += (j & 1) ? 2 * G - 1 : 1) {   // the pairs of points g, g + G, ...
            const cpx<T> u = buf[K::s_pos(j)];
            const double x = u.x, y = u.y;
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

    // The potential factor and a norm sum that tells a non-finite state (there are no jumps, so nothing else is
    // done with it and the sum leaves out the weight |K_V|^2, an expf a point):
    // mode 0: x <- stat1 dyn_b x (the first half-step of a trajectory)
    // mode 1: x <- stat2 dyn_a dyn_b x; returns sum |x_old|^2
    // mode 2: x <- stat1 dyn_a x; returns sum |x_new|^2
    // The dynamic exponent of the half-step at temperature T is (V_I - i (V_R + a/r)) dt/2 at each point, evaluated
    // per point and applied as w + w f1 (fused.cuh); ka, kb are the per-step scalars of T_n (the closing half-step)
    // and T_{n+1} (the opening one).
    // CACHE: the potential at T_{n+1} is kept in shared memory (vc, thread-private places) for the next step's T_n.
    // (Of the even points alone it fits at N = 4096 too, but the L1 that this takes made the step 20% slower.)
    // The loop is not unrolled: with two pairs of points in flight the code outgrows the instruction cache once the CTAs
    // have drifted apart (N = 4096 through 2404 steps: 1.15e7 trajectory-steps/s unrolled, 1.25e7 not; 1.21e7 before the
    // norm's weight was left out; N = 1024: 5.95e7, 6.54e7, 4.87e7).
    template <bool CACHE>
    static __device__ typename NormSum<T>::type factor_ksu(cpx<T> *buf, const Tables<T> &tb, int g, int l, int mode,
                                                           const KsuT<T> &ka, const KsuT<T> &kb, float2 *vc, double *red)
    {
        SqAcc<T> acc, acc_odd;
        const SC *tab = (mode == 1) ? tb.statV2 : tb.statV;
        const T hdt = (T)0.5 * tb.ksu_dt;
#pragma unroll 1
        for (int k = g; k < N / 2; k += G) {
#pragma unroll
            for (int par = 0; par < 2; ++par) {
                const int j = 2 * k + par;
                const int p = par ? K::odd_pos(k) : K::even_pos(k);
                const T fj = (T)j;
                T A = (T)0, t = (T)0;
                if (j > 0) {
                    T vda = (T)0, via = (T)0, vdb = (T)0, vib = (T)0;
                    if constexpr (CACHE) {
                        float2 *q = vc + par * (N / 2) + k;
                        if (mode != 0) {
                            vda = q->x;
                            via = q->y;
                        }
                        if (mode != 2) {
                            ksu_point<T>(tb, kb, fj, vdb, vib);
                            *q = make_float2(vdb, vib);
                        }
                    } else {
                        if (mode != 0) ksu_point<T>(tb, ka, fj, vda, via);
                        if (mode != 2) ksu_point<T>(tb, kb, fj, vdb, vib);
                    }
                    A = (via + vib) * hdt;
                    t = -(vda + vdb) * hdt;
                }
                T f1r, f1i, em1;
                Dyn<T>::f1t(A, t, &f1r, &f1i, &em1);
                cpx<T> v = buf[p];
                SqAcc<T> &ac = par ? acc_odd : acc;
                if (mode == 1) ac.add_w(v, (T)1);
                const cpx<T> w = PR::mul_s(v, stat(tb, tab, 0, l, j, mode == 1));
                v = mk(w.x + (w.x * f1r - w.y * f1i), w.y + (w.x * f1i + w.y * f1r));
                if (mode == 2) ac.add_w(v, (T)1);
                buf[p] = v;
            }
        }
        if (mode == 0) return {};
        acc.merge(acc_odd);
        return slot_norm_sum<T, G>(acc, red);
    }
};

template <int N>
__global__ void __launch_bounds__(NftPlan<N>::G, (NftPlan<N>::MIN_BLOCKS)) ksu32_kernel(Tables<float> tb, LaunchArgs a)
{
    using T = float;
    using K = NftSine<N>;
    using PW = NftPointwise<N>;
    constexpr int G = K::G, E = K::E;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cpx<T> *buf = reinterpret_cast<cpx<T> *>(smem_raw);
    using C = typename Prec<T>::C;
    using P = NftPlan<N>;
    C *tw1 = reinterpret_cast<C *>(buf + P::BUF);
    C *tw2 = tw1 + P::TW1;
    Carry *wtot = reinterpret_cast<Carry *>(tw2 + P::TW2);
    double *red = reinterpret_cast<double *>(wtot + (G / 32 + 1)), *fin = red + 8 * (G / 32 + 1);
    float2 *vc = reinterpret_cast<float2 *>(fin + 8);
    __shared__ int s_traj;
    // middle-pass twiddles, row m of a table holding W^(m k) for every k (tw1: [M1][R] of W_{R M1},
    // tw2: [M2][R M1] of W_{R M1 M2}, the second only with a second middle pass), built once per CTA
    for (int t = threadIdx.x; t < P::TW1; t += G)
        tw1[t] = Prec<T>::ld(&tb.W[(t / P::R) * (t % P::R) * (N / P::TW1)]);
    if (P::M2 > 1)
        for (int t = threadIdx.x; t < P::TW2; t += G)
            tw2[t] = Prec<T>::ld(&tb.W[(t / P::TW1) * (t % P::TW1) * (N / P::TW2)]);

    const int g = threadIdx.x;
    const double dr = tb.dr;
    cpx<T> x[E];

    for (;;) {
        if (g == 0) s_traj = fetch_trajectory(tb, a);
        __syncthreads();
        const int t = s_traj;
        __syncthreads();
        if (t < 0) break;
        const TrajDev d = a.trajs[t];
        const MediumDev md = tb.media[d.medium];
        const int l = tb.spec_l[d.spec];
        const double *ic = tb.ic + (size_t)d.spec * N;
        for (int k = g; k < N / 2; k += G) {
            buf[K::even_pos(k)] = mk<T>((T)ic[2 * k], (T)0);
            buf[K::odd_pos(k)] = mk<T>((T)ic[2 * k + 1], (T)0);
        }
        Threshold<T> thr;
        thr.set(-1.0, dr);
        int flags = 0, ended = 0, executed = 0;
        const int ns = d.n_steps;
        const T mA = (T)md.A, mtau0 = (T)md.tau0, mdtau = (T)md.dtau;
        int seg = 0;
        auto T3_of = [&](int n) -> T {
            return md.kind == 1 ? table_T3_far<T>(tb.prof + 2 * (size_t)md.tab_off, md.tab_len, mtau0 + (T)n * mdtau, &seg)
                                : mA / (mtau0 + (T)n * mdtau);
        };
        T T3b = T3_of(0);
        KsuT<T> kb = ksu_at<T>(tb, T3b);
        if (ns > 0) {
            __syncthreads();
            PW::template factor_ksu<P::CACHE>(buf, tb, g, l, 0, kb, kb, vc, red);
        }
        for (int n = 0; n < ns; ++n) {
            const bool last = (n + 1 == ns);
            T3b = T3_of(n + 1);
            __syncthreads();
#pragma unroll 1
            for (int h = 0; h < 2; ++h) K::dst(x, buf, tb, g, wtot, tw1, tw2, h == 1);
            executed = n + 1;
            const KsuT<T> ka = kb;
            kb = ksu_at<T>(tb, T3b);
            const typename NormSum<T>::type n2s = PW::template factor_ksu<P::CACHE>(buf, tb, g, l, last ? 2 : 1, ka, kb, vc, red);
            if (!thr.finite(n2s)) {
                flags |= QTRAJ_F_NONFINITE;
                ended = 1;
                if (g == 0) atomicOr(a.status, 1);
                break;
            }
        }
        __syncthreads();

        // the norm and the overlaps as fused.cuh's read-out; without jumps the norm lost to V_I is the dissociation, and
        // the overlap is taken unnormalised
        const int nb = ended || l > 2 ? 0 : 3 - l;
        auto state_of = [&](int i) { return l == 0 ? (i == 2 ? 3 : i) : l == 1 ? 2 + 2 * i : 5; };
        {
            Dot2 norm, dot[3];
            for (int k = g; k < N / 2; k += G) {
                const cpx<T> a0 = buf[K::even_pos(k)], a1 = buf[K::odd_pos(k)];
                const float2 u0 = make_float2(a0.x, a0.y), u1 = make_float2(a1.x, a1.y);
                norm.add(u0, u0);
                norm.add(u1, u1);
#pragma unroll
                for (int i = 0; i < 3; ++i)
                    if (i < nb) {
                        const float4 f = __ldg(reinterpret_cast<const float4 *>(tb.eigo + (size_t)state_of(i) * N) + k);
                        dot[i].add(Prec<float>::Rl{f.x, f.y}, u0);
                        dot[i].add(Prec<float>::Rl{f.z, f.w}, u1);
                    }
            }
            double v[8] = {norm.x() + norm.y(), dot[0].x(), dot[0].y(), dot[1].x(), dot[1].y(), dot[2].x(), dot[2].y(), 0};
            slot_sums8<G>(v, red, fin);
            traj_sync<G>();
            if (ns == 0 || !dot2_holds(fin[0])) PW::read_out64(buf, tb, g, nb, l, red, fin);
        }
        if (a.states) {
            double *st = a.states + (size_t)t * N * 2;
            for (int k = g; k < N / 2; k += G) {
                const cpx<T> a0 = buf[K::even_pos(k)], a1 = buf[K::odd_pos(k)];
                st[4 * k] = (double)a0.x;
                st[4 * k + 1] = (double)a0.y;
                st[4 * k + 2] = (double)a1.x;
                st[4 * k + 3] = (double)a1.y;
            }
        }
        if (g < 32) {
            qtraj_obs *o = a.obs + t;
            for (int q = g; q < NBASIS; q += G < 32 ? G : 32) {
                const int ql = q == 2 || q == 4 ? 1 : q == 5 ? 2 : 0, i = q < 3 ? (q == 2 ? 0 : q) : q == 3 ? 2 : q == 4 ? 1 : 0;
                double re = 0.0, im = 0.0, sv = 0.0;
                if (nb > 0 && ql == l) {
                    re = fin[1 + 2 * i] * dr;
                    im = fin[2 + 2 * i] * dr;
                    sv = re * re + im * im;
                    if (!tb.ov0_zero[d.spec * NBASIS + q]) {
                        const double a0 = tb.ov0[(d.spec * NBASIS + q) * 2], b0 = tb.ov0[(d.spec * NBASIS + q) * 2 + 1];
                        sv /= a0 * a0 + b0 * b0;
                    }
                }
                o->surv[q] = sv;
                o->ov_re[q] = re;
                o->ov_im[q] = im;
            }
            if (g == 0) {
                o->norm2 = fin[0] * dr;
                o->r0 = 0.0;
                o->l = l;
                o->color = 0;
                o->n_jumps = 0;
                o->n_steps_exec = executed;
                o->flags = flags;
                o->first_jump_step = -1;
                o->last_jump_step = -1;
                o->jump_digest = DIGEST_BASIS;
            }
        }
        __syncthreads();
    }
}

// launches ksu32_kernel<N> (fused_go)
template <int N>
cudaError_t ksu32_go(const Tables<float> &tb, const LaunchArgs &a, int sm_count, int max_ctas, cudaStream_t s,
                     FusedInfo *info, bool query_only)
{
    using P = NftPlan<N>;
    constexpr int smem = P::SMEM + (P::CACHE ? N * 8 : 0);
    return launch_wave(ksu32_kernel<N>, P::G, P::R, smem, tb, a, sm_count, max_ctas, s, info, query_only);
}

} // namespace qt
