// plain.cu -- the plain per-step FP64 form (plain.cuh): set-up, waiting-time test and jump, read-out, and the step
// loop on the host.
#include "plain.cuh"

namespace qt {

namespace {

constexpr int PB = 256; // threads of the per-trajectory kernels

// the state's layout (PlainBuffers): grid point of the value at i, and its sign
struct Order {
    int R, M, G;
    __device__ __forceinline__ int j(int i) const { return plan_j(i % G, i / G, R, M, G); }
    __device__ __forceinline__ double sign(int i) const { return i / G % R < R / 2 ? 1.0 : -1.0; }
};

// block-wide sum of a double over PB threads, same value returned to every thread
__device__ double block_sum(double v, double *sh)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    for (int w = 0; w < PB / 32; ++w) s += sh[w];
    __syncthreads();
    return s;
}

__global__ void plain_setup(Tables<double> tb, LaunchArgs a, PlainState *st, cpx<double> *psi, int N, Order ord)
{
    const int b = blockIdx.x;
    __shared__ int s_active;
    const TrajDev d = a.trajs[b];
    if (threadIdx.x == 0) {
        PlainState s;
        const Draws dw = draws(d.seed, 0u);
        s.thr = a.nojump ? -1.0 : dw.r;
        s.ul = dw.ul;
        s.uc = dw.uc;
        s.r0 = a.nojump ? 0.0 : dw.r;
        s.l = tb.spec_l[d.spec];
        s.c = tb.spec_color[d.spec];
        s.nj = 0;
        s.fj = -1;
        s.flags = 0;
        s.active = 1;
        s.kdraw = 0;
        s.executed = 0;
        s.lj = -1;
        s.digest = DIGEST_BASIS;
        if (!a.nojump) {
            if (tb.use_rmin) {
                const qtraj_obs &gj = a.group[d.group];
                if (fabs(dw.r - gj.norm2) < BORDER_EPS) s.flags |= QTRAJ_F_BORDERLINE;
                if (dw.r < gj.norm2) {
                    qtraj_obs o = gj;
                    o.r0 = dw.r;
                    o.n_steps_exec = 0;
                    o.flags = s.flags | QTRAJ_F_NOJUMP_SHORTCUT;
                    a.obs[b] = o;
                    s.active = 0;
                }
            }
            if (s.active && dw.r > tb.r_max) {
                qtraj_obs o;
                for (int q = 0; q < NBASIS; ++q) { o.surv[q] = 0; o.ov_re[q] = 0; o.ov_im[q] = 0; }
                o.norm2 = 1.0;
                o.r0 = dw.r;
                o.l = s.l;
                o.color = s.c;
                o.n_jumps = 0;
                o.n_steps_exec = 0;
                o.flags = s.flags | QTRAJ_F_RMAX;
                o.first_jump_step = -1;
                o.last_jump_step = -1;
                o.jump_digest = DIGEST_BASIS;
                a.obs[b] = o;
                s.active = 0;
            }
        }
        if (s.active && d.n_steps == 0) s.active = 2;   // finalised by plain_finalize_empty
        st[b] = s;
        s_active = s.active;
    }
    __syncthreads();
    if (s_active) {
        const double *ic = tb.ic + (size_t)d.spec * N * (tb.ic_cplx ? 2 : 1);
        for (int i = threadIdx.x; i < N; i += blockDim.x) {
            const int j = ord.j(i);
            const double sg = ord.sign(i);
            psi[(size_t)b * N + i] = tb.ic_cplx ? mk(sg * ic[2 * j], sg * ic[2 * j + 1]) : mk(sg * ic[j], 0.0);
        }
    }
}

__device__ void plain_write_obs(const Tables<double> &tb, const LaunchArgs &a, int b, const TrajDev &d,
                                const PlainState &s, const cpx<double> *p, int N, Order ord, int ended, double *sh)
{
    const int basis_l[NBASIS] = {0, 0, 1, 0, 1, 2};
    double acc = 0.0;
    for (int j = threadIdx.x; j < N; j += PB) acc = fma(p[j].x, p[j].x, fma(p[j].y, p[j].y, acc));
    const double n2 = block_sum(acc, sh) * tb.dr;
    double ovr[NBASIS], ovi[NBASIS];
    for (int q = 0; q < NBASIS; ++q) {
        ovr[q] = 0.0;
        ovi[q] = 0.0;
        if (ended || s.c != 0 || basis_l[q] != s.l) continue;
        const double *phi = tb.eig + (size_t)q * N;
        double pr = 0.0, pi = 0.0;
        for (int i = threadIdx.x; i < N; i += PB) {
            const double f = ord.sign(i) * phi[ord.j(i)];
            pr += f * p[i].x;
            pi += f * p[i].y;
        }
        ovr[q] = block_sum(pr, sh) * tb.dr;
        ovi[q] = block_sum(pi, sh) * tb.dr;
    }
    if (a.states) {
        double *out = a.states + (size_t)b * N * 2;
        for (int i = threadIdx.x; i < N; i += PB) {
            const int j = ord.j(i);
            const double sg = ord.sign(i);
            out[2 * j] = sg * p[i].x;
            out[2 * j + 1] = sg * p[i].y;
        }
    }
    if (threadIdx.x == 0) {
        qtraj_obs o;
        for (int q = 0; q < NBASIS; ++q) {
            o.ov_re[q] = ovr[q];
            o.ov_im[q] = ovi[q];
            double sv = 0.0;
            if (!ended && s.c == 0 && basis_l[q] == s.l) {
                const double prob = (ovr[q] * ovr[q] + ovi[q] * ovi[q]) / n2;
                if (tb.ov0_zero[d.spec * NBASIS + q]) sv = prob;
                else {
                    const double a0 = tb.ov0[(d.spec * NBASIS + q) * 2], b0 = tb.ov0[(d.spec * NBASIS + q) * 2 + 1];
                    sv = prob / (a0 * a0 + b0 * b0);
                }
            }
            o.surv[q] = sv;
        }
        o.norm2 = n2;
        o.r0 = s.r0;
        o.l = s.l;
        o.color = s.c;
        o.n_jumps = s.nj;
        o.n_steps_exec = s.executed;
        o.flags = s.flags;
        o.first_jump_step = s.fj;
        o.last_jump_step = s.lj;
        o.jump_digest = s.digest;
        a.obs[b] = o;
    }
}

// waiting-time test after step n, the jump, and the read-out after the last step (Sec. 3.5 item 4)
__global__ void __launch_bounds__(PB) plain_jump(Tables<double> tb, LaunchArgs a, PlainState *st, cpx<double> *psi,
                                                 const double *n2in, int parts, int N, Order ord, int n)
{
    const int b = blockIdx.x;
    const TrajDev d = a.trajs[b];
    PlainState s = st[b];
    if (!plain_running(s, d, n)) return;
    __shared__ double sh[PB / 32];
    cpx<double> *p = psi + (size_t)b * N;
    double n2 = 0.0;
    for (int i = 0; i < parts; ++i) n2 += n2in[(size_t)b * parts + i];
    n2 *= tb.dr;
    s.executed = n + 1;
    int ended = 0, jump = 0;
    int l_new = s.l, c_new = s.c;
    if (!isfinite(n2)) {
        s.flags |= QTRAJ_F_NONFINITE;
        ended = 1;
        if (threadIdx.x == 0) atomicOr(a.status, 1);
    } else if (!a.nojump) {
        if (fabs(n2 - s.thr) < BORDER_EPS) s.flags |= QTRAJ_F_BORDERLINE;
        if (n2 <= s.thr) {
            if (tb.max_jumps >= 0 && s.nj >= tb.max_jumps) {
                s.flags |= QTRAJ_F_MAXJUMPS;
                ended = 1;
            } else {
                l_new = (s.ul < (double)s.l / (2.0 * s.l + 1.0)) ? s.l - 1 : s.l + 1;
                c_new = (s.c == 1 && s.uc < tb.p_os) ? 0 : 1;
                if (s.fj < 0) s.fj = n;
                if (tb.l_cap >= 0 && l_new > tb.l_cap) {
                    s.flags |= QTRAJ_F_LCAP;
                    s.l = l_new;
                    s.c = c_new;
                    ++s.nj;
                    s.lj = n;
                    s.digest = digest_jump(s.digest, n, s.l, s.c);
                    ended = 1;
                } else {
                    jump = 1;
                }
            }
        }
    }
    if (jump) {
        double acc = 0.0;
        for (int i = threadIdx.x; i < N; i += PB) {
            const double rj = ord.j(i) * tb.dr;
            const cpx<double> v = scale(p[i], rj);
            p[i] = v;
            acc = fma(v.x, v.x, fma(v.y, v.y, acc));
        }
        const double tot = block_sum(acc, sh) * tb.dr;
        const double inv = 1.0 / sqrt(tot);
        for (int j = threadIdx.x; j < N; j += PB) p[j] = scale(p[j], inv);
        __syncthreads();
        s.l = l_new;
        s.c = c_new;
        ++s.nj;
        s.lj = n;
        s.digest = digest_jump(s.digest, n, s.l, s.c);
        ++s.kdraw;
        const Draws dw = draws(d.seed, (uint32_t)s.kdraw);
        s.thr = dw.r;
        s.ul = dw.ul;
        s.uc = dw.uc;
    }
    if (ended || n == d.n_steps - 1) {
        plain_write_obs(tb, a, b, d, s, p, N, ord, ended, sh);
        s.active = 0;
    }
    if (threadIdx.x == 0) st[b] = s;
}

// trajectories whose medium has no step at all (T0 <= Tf) are read out unevolved
__global__ void __launch_bounds__(PB) plain_finalize_empty(Tables<double> tb, LaunchArgs a, PlainState *st,
                                                           const cpx<double> *psi, int N, Order ord)
{
    const int b = blockIdx.x;
    PlainState s = st[b];
    if (s.active != 2) return;
    __shared__ double sh[PB / 32];
    plain_write_obs(tb, a, b, a.trajs[b], s, psi + (size_t)b * N, N, ord, 0, sh);
    if (threadIdx.x == 0) { s.active = 0; st[b] = s; }
}

} // namespace

static const PlainOps *ops_of(int N) { return N <= 2048 ? plain_ops_a(N) : plain_ops_b(N); }
size_t plain_seq(int N) { return (size_t)ops_of(N)->seq; }
int plain_parts(int N) { return ops_of(N)->parts; }

cudaError_t plain_run(const Tables<double> &tb, const LaunchArgs &a, int N, int max_steps, PlainBuffers buf,
                      cudaStream_t stream, int *launches)
{
    const int B = a.n_traj;
    if (B == 0) return cudaSuccess;
    const PlainOps *ops = ops_of(N);
    const Plan p = make_plan(N, true, PLAN_PLAIN);
    const Order ord{p.R, p.M, p.G};
    plain_setup<<<B, PB, 0, stream>>>(tb, a, buf.st, buf.psi, N, ord);
    plain_finalize_empty<<<B, PB, 0, stream>>>(tb, a, buf.st, buf.psi, N, ord);
    for (int n = 0; n < max_steps; ++n) {
        const cudaError_t e = ops->step(tb, a, buf, n, stream);
        if (e != cudaSuccess) return e;
        plain_jump<<<B, PB, 0, stream>>>(tb, a, buf.st, buf.psi, buf.n2, ops->parts, N, ord, n);
    }
    if (launches) *launches += 2 + 6 * max_steps;
    return cudaGetLastError();
}

} // namespace qt
