// plain_step.cuh -- the five transform kernels of a step of the plain form (plain.cuh), for one grid size.
//
// A step through separate FFT passes of radix 4 took 18 kernels, each a pass over the batch's states (750 us at N =
// 16384, 40 trajectories, where the FP64 work fills 100 us).  The radices 32 x 32 x 32 of the fused plan leave three
// passes a transform, and the pointwise factors ride on the last and first ones.  Blocks of one warp (32 slots of R
// values): the FP64 pipe of an SM quarter is busy with one warp, and small blocks spread evenly over the SMs.
#pragma once
#include "fused.cuh"
#include "plain.cuh"

namespace qt {

template <int N> struct PlainStep {
    using P = FusedPlan<double, N, 7>;
    using K = Sine<double, N, 7>;
    using PW = Pointwise<double, N, 7>;
    using PR = Prec<double>;
    static constexpr int G = P::G, E = P::E, R = P::R, H = P::H, M = P::M, S = P::S, NS = P::NS;
    static constexpr int TB = G < 32 ? G : 32, NB = G / TB;   // threads of a block, blocks of a trajectory
    static_assert(P::M2 == 1 && M <= 32, "one middle pass; split() inside a warp");

    // the block's trajectory and the thread's place in it
    struct Place {
        int b, g, pb[NS], pm[NS];
        __device__ __forceinline__ Place() : b((int)blockIdx.x / NB), g((int)(blockIdx.x % NB) * TB + threadIdx.x)
        {
#pragma unroll
            for (int t = 0; t < NS; ++t) {
                int lo, hi;
                slot_points(g + t * G, R, M, lo, hi);
                pb[t] = K::pos(lo);
                pm[t] = K::pos(S - lo);
            }
        }
    };

    // x <- K_V(n) x, a half-step; returns sum |x|^2 of the thread's values
    static __device__ __forceinline__ double half_step(cpx<double> *x, const Tables<double> &tb, const MediumDev &md, int c,
                                                       int l, int n, int g)
    {
        const double tau = md.tau0 + (double)n * md.dtau;
        const double T3 = md.kind == 1 ? table_T3_at(tb.prof + 2 * (size_t)md.tab_off, md.tab_len, tau) : md.A / tau;
        const double A = md.erj[c] * kappa_T3<double>(md.kfit, T3), B = 3.14159265358979323846 * md.eij[c] * T3;
        const cpx<double> *row = tb.statV + ((size_t)c * LTAB + l) * N;
        double qw, sum = 0.0;
        const cpx<double> qe = Dyn<double>::cexp<true>(2.0 * A * S * S, 2.0 * B * S * S, &qw);
#pragma unroll
        for (int t = 0; t < NS; ++t) {
            int lo, hi;
            slot_points(g + t * G, R, M, lo, hi);
            typename PW::Run ul, uh;
            ul.template start<true>(A, B, 0.0, (double)lo);
            uh.template start<true>(A, B, 0.0, (double)hi);
#pragma unroll
            for (int m = 0; m < H; ++m) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    typename PW::Run &u = h ? uh : ul;
                    const int e = t * R + (h ? R - 1 - m : m);
                    const cpx<double> s = l < LTAB ? PR::ld_s(row + PW::stat_idx(g, e)) : PW::stat(tb, tb.statV, c, l, g, e, false);
                    x[e] = PR::mul_s(x[e], s) * u.e;
                    sum = fma(x[e].x, x[e].x, fma(x[e].y, x[e].y, sum));
                    if (m + 1 < H) u.template step<true>(qe, qw);
                }
            }
        }
        return sum;
    }

    static __device__ __forceinline__ bool off(const LaunchArgs &a, const PlainState *st, int b, int n)
    {
        return b >= a.n_traj || !plain_running(st[b], a.trajs[b], n);
    }
};

// start of step n: the first pass of K_V psi
template <int N>
__global__ void __launch_bounds__(PlainStep<N>::TB) plain_first(Tables<double> tb, LaunchArgs a, PlainBuffers buf, int n)
{
    using L = PlainStep<N>;
    const typename L::Place p;
    if (L::off(a, buf.st, p.b, n)) return;
    cpx<double> x[L::P::XN];
    const cpx<double> *psi = buf.psi + (size_t)p.b * N;
#pragma unroll
    for (int e = 0; e < L::E; ++e) x[e] = psi[e * L::G + p.g];
    L::half_step(x, tb, tb.media[a.trajs[p.b].medium], buf.st[p.b].c, buf.st[p.b].l, n, p.g);
    L::K::first(x, buf.sa + (size_t)p.b * L::P::BUF, tb.TA, tb.TH, p.g, p.pb, p.pm);
}

template <int N>
__global__ void __launch_bounds__(PlainStep<N>::TB) plain_mid(Tables<double> tb, LaunchArgs a, PlainBuffers buf, cpx<double> *s, int n)
{
    using L = PlainStep<N>;
    const typename L::Place p;
    if (L::off(a, buf.st, p.b, n)) return;
    cpx<double> x[L::P::XN];
    L::K::mid(x, s + (size_t)p.b * L::P::BUF, tb.TM, tb.TI, tb.TS, p.g);
}

// between the transforms: last pass, kinetic factor, first pass
template <int N>
__global__ void __launch_bounds__(PlainStep<N>::TB) plain_kinetic(Tables<double> tb, LaunchArgs a, PlainBuffers buf, int n)
{
    using L = PlainStep<N>;
    const typename L::Place p;
    if (L::off(a, buf.st, p.b, n)) return;
    cpx<double> x[L::P::XN];
    L::K::last(x, buf.sa + (size_t)p.b * L::P::BUF, tb.TM, p.g);
    L::K::kinetic(x, tb.KF, p.g);
    L::K::first(x, buf.sb + (size_t)p.b * L::P::BUF, tb.TA, tb.TH, p.g, p.pb, p.pm);
}

// end of the step: last pass, space half-step, the block's part of the norm
template <int N>
__global__ void __launch_bounds__(PlainStep<N>::TB) plain_last(Tables<double> tb, LaunchArgs a, PlainBuffers buf, int n)
{
    using L = PlainStep<N>;
    const typename L::Place p;
    if (L::off(a, buf.st, p.b, n)) return;
    cpx<double> x[L::P::XN];
    L::K::last(x, buf.sb + (size_t)p.b * L::P::BUF, tb.TM, p.g);
    double v = L::half_step(x, tb, tb.media[a.trajs[p.b].medium], buf.st[p.b].c, buf.st[p.b].l, n, p.g);
    cpx<double> *psi = buf.psi + (size_t)p.b * N;
#pragma unroll
    for (int e = 0; e < L::E; ++e) psi[e * L::G + p.g] = x[e];
#pragma unroll
    for (int off = L::TB / 2; off > 0; off >>= 1) v += __shfl_xor_sync(lane_mask<L::TB>(), v, off, L::TB);
    if (threadIdx.x == 0) buf.n2[blockIdx.x] = v;
}

template <int N> cudaError_t plain_step(const Tables<double> &tb, const LaunchArgs &a, PlainBuffers buf, int n, cudaStream_t s)
{
    using L = PlainStep<N>;
    const int blocks = a.n_traj * L::NB;
    plain_first<N><<<blocks, L::TB, 0, s>>>(tb, a, buf, n);
    plain_mid<N><<<blocks, L::TB, 0, s>>>(tb, a, buf, buf.sa, n);
    plain_kinetic<N><<<blocks, L::TB, 0, s>>>(tb, a, buf, n);
    plain_mid<N><<<blocks, L::TB, 0, s>>>(tb, a, buf, buf.sb, n);
    plain_last<N><<<blocks, L::TB, 0, s>>>(tb, a, buf, n);
    return cudaGetLastError();
}

template <int N> const PlainOps *plain_ops()
{
    static const PlainOps ops = {PlainStep<N>::P::BUF, PlainStep<N>::NB, plain_step<N>};
    return &ops;
}

} // namespace qt
