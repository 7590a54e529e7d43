// fused_plan.h -- the decomposition of the fused kernel's sine transform for every grid size, shared by
// the kernel and by the host code that lays its tables out.
//
// The DST-I of N points is the length-2N FFT of the odd extension, done as a radix-R pass, a middle
// transform of M = 2N/R^2 points (one pass M1, or two passes M1 x M2) and a radix-R pass, of which only
// the half that the odd symmetry leaves independent is computed (fused.cuh).  The state lives in registers
// as N/R "slots" of R values; slot s, value m is the grid point
//     j = lo + S m (m < R/2),   hi + S (R-1-m) (m >= R/2),      S = 2N/R = R M,
// whose register holds u_j for m < R/2 and -u_j for m >= R/2 (the odd extension at lo + S m).  Thread g of
// G = N/E holds the slots g, g + G, ... (E/R of them).
#pragma once
#include <cuda_runtime.h>

namespace qt {

struct PlanDims { int R, E, M1, M2; };

// The plans.  FP32 up to N = 4096: 16 values a thread where two warps of a trajectory then share an SM quarter and its
// instruction fetch, 32 above (fewer exchanges).  FP64: 4 to 32 values a thread.  An FP64 instruction takes a warp 64
// cycles whatever its lanes do and an SM completes one every 19, so a few FP64 trajectories want four warps with little
// each, and a full device few instructions; the plans up to N = 1024 are those of the shorter step (us a step of 8
// trajectories / 10^6 trajectory-steps a second of 3000): N = 1024 radix 8, 8 x 4 44.4 / 3.9, radix 16, 8 65.7 / 4.6;
// FP32 N = 128 radix 4, 16 2.2 / 642, radix 8, 4 2.9 / 602.
// The share of the spectrum that goes through a running sum, 2/R, sets the rounding noise: FP64 N = 256 and 512 keep radix 8
// for it.  Radix 4, 4 x 8 at N = 256 left final states 5.8e-14 off after 64 steps where the earlier transform left
// 3.4e-14 (radix 8 1.6e-14); radix 4, 8 x 8 at N = 512 left 2.5e-14 after 4 steps (earlier transform 0.9e-14; radix 8,
// 8 x 2 0.6e-14; radix 8, 16 0.4e-14; a step of 8 trajectories 29.5, 37.9 and 41.8 us, 300 steps of 3000 58.0, 61.3 and
// 58.7 ms; a full wave without jumps 7.4e6 trajectory-steps/s with radix 4, 8.5e6 with 8 x 2).  FP32 at N = 256 and above keeps the larger radix, for the noise and for the throughput (N = 512 radix 8,
// 16 2.9 / 226, radix 16, 4 4.2 / 284).
// RAD8: the radix-8 plans of the launch variants 2 and 3 (FP32, N = 2048 and 4096); PLAIN: the plain form's, one
// middle pass and at most 32 of a sequence's slots (plain_step.cuh).
enum PlanKind { PLAN_FUSED = 0, PLAN_RAD8 = 1, PLAN_PLAIN = 2 };
__host__ __device__ constexpr PlanDims plan_dims(int N, bool f64, PlanKind kind)
{
    if (kind == PLAN_RAD8 && !f64 && N == 2048) return {8, 16, 8, 8};
    if (kind == PLAN_RAD8 && !f64 && N == 4096) return {8, 16, 16, 8};
    if (f64 && kind != PLAN_PLAIN) {
        switch (N) {
        case 128: return {4, 4, 4, 4};
        case 512: return {8, 8, 8, 2};
        case 1024: return {8, 8, 8, 4};
        default: break;
        }
    }
    switch (N) {
    case 16: return {4, 4, 2, 1};
    case 32: return {4, 4, 4, 1};
    case 64: return {4, 4, 8, 1};
    case 128: return {4, 4, 16, 1};
    case 256: return {8, 8, 8, 1};
    case 512: return f64 ? PlanDims{8, 8, 16, 1} : PlanDims{16, 16, 4, 1};
    case 1024: return {16, 16, 8, 1};
    case 2048: return {16, 16, 16, 1};
    case 4096: return f64 ? PlanDims{16, 32, 32, 1} : PlanDims{16, 16, 32, 1};
    case 8192: return {32, 32, 16, 1};
    default: return {32, 32, 32, 1};   // 16384
    }
}

// The slot's base points.  Slot s = kk M + q1 belongs to the residue b = kk + R q1 modulo S and holds the
// points j = +-b (mod S).  kk = 0 holds the residues 0 and R/2 modulo R: q1 = 0 the points that are
// multiples of S/2 (two half-length sequences in one slot), 0 < q1 < M/2 the residue R q1, and
// q1 >= M/2 the residue R/2 + R q1.
__host__ __device__ __forceinline__ void slot_points(int s, int R, int M, int &lo, int &hi)
{
    const int S = R * M, kk = s / M, q1 = s % M;
    if (s == 0) {
        lo = 0;
        hi = S / 2;
        return;
    }
    const int b = kk ? kk + R * q1 : (q1 < M / 2 ? R * q1 : R / 2 + R * q1);
    lo = b;
    hi = S - b;
}

// grid point of element e (slot e / R of thread g, value e % R)
__host__ __device__ __forceinline__ int plan_j(int g, int e, int R, int M, int G)
{
    int lo, hi;
    slot_points(g + (e / R) * G, R, M, lo, hi);
    const int m = e % R;
    return m < R / 2 ? lo + R * M * m : hi + R * M * (R - 1 - m);
}

// Tables with one entry per grid point are laid out in the order the threads read them: the pair of
// elements (m, R-1-m) of a slot together, threads side by side.  16-byte entries (kinetic factors, FP64
// static factors): two rows of G entries per pair; 8-byte entries (FP32 static factors): the two entries
// of a thread's pair adjacent, one 16-byte load.  Element e of the entry at index i of thread g:
__host__ __device__ __forceinline__ void plan_entry(int i, bool adjacent, int R, int G, int &g, int &e)
{
    int pr, h;
    if (adjacent) {
        pr = i / 2 / G;
        g = i / 2 % G;
        h = i & 1;
    } else {
        pr = i / (2 * G);
        h = i / G % 2;
        g = i % G;
    }
    const int t = pr / (R / 2), m = pr % (R / 2);
    e = t * R + (h ? R - 1 - m : m);
}

// The FP32 KSU kernel's radix (fused_ksu32.cuh), and the radix of its compact last-pass twiddle table, which it reads up
// to N = 2048 (0: none)
__host__ __device__ constexpr int ksu32_radix(int N) { return N <= 32 ? 4 : N <= 2048 ? 8 : 16; }
__host__ __device__ constexpr int ksu32_wl_radix(int N) { return N <= 2048 ? ksu32_radix(N) : 0; }

// host view of a plan
struct Plan {
    int N, R, E, M, M1, M2, G, S, NS;
    bool tw_last;   // W_S^{b1 q1} is applied by the last pass (else by the middle one)
};
__host__ __device__ constexpr bool plan_tw_last(PlanDims d) { return d.M2 > 1 || d.M1 >= d.R; }
inline Plan make_plan(int N, bool f64, PlanKind kind)
{
    const PlanDims d = plan_dims(N, f64, kind);
    const int M = d.M1 * d.M2;
    return {N, d.R, d.E, M, d.M1, d.M2, N / d.E, d.R * M, N / d.R, plan_tw_last(d)};
}

} // namespace qt
