"""Inputs at the ends of their ranges: states decayed below FP32's products, temperatures that drop within a step,
exponents beyond FP32's, and repeated calls that may not wait for each other."""
import numpy as np
import pytest

from test_gpu_parity import check_fp32, check_fp64, fp32_bound, oracle_inputs, q, run_gpu, run_oracle  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("potential", [0, 1])
def test_fp32_read_out_of_decayed_states(q, potential):  # noqa: F811
    """No-jump evolutions whose norm falls to 1e-26 .. 1e-53, where squares of the FP32 amplitudes underflow: norms
    and ratios as the FP64 form's, within the FP32 state's error (norm and ratio are quadratic in it)."""
    import torch
    if potential:
        N, L, dt, med = 64, 12.0, 0.05, q.medium(2.0, 25.0, 1.5, 0.0, 0.0)
    else:
        N, L, dt, med = 64, 6.0, 0.01, q.medium(0.6, 0.6, 0.3, 100.0, -1.0)
    res = []
    for prec in (q.FP64, q.FP32):
        e = q.Engine(q.Config(N=N, L=L, dt=dt, precision=prec, potential=potential))
        e.init([q.init_spec("gauss", 0.8, 1, 0, 0), q.init_spec("gauss", 0.8, 2, 1, 0)], 2, np.arange(2))
        e.evolve([med], np.arange(2, dtype=np.uint64))
        o = e.observables(check_finite=False)
        torch.cuda.synchronize()
        res.append(o if potential else e.nojump_results(2))   # (OQS: the groups' no-jump records)
        e.close()
    a, b = res
    assert (a["norm2"] > 0).all() and a["norm2"].min() < 1e-45 and (a["n_steps_exec"] > 1000).all()
    bound = 2 * fp32_bound(N, a["n_steps_exec"])
    assert (np.abs(b["norm2"] / a["norm2"] - 1) <= bound).all(), (a["norm2"], b["norm2"])
    top = a["surv"].max(1)
    assert np.isfinite(b["surv"]).all() and (np.abs(b["surv"] - a["surv"]).max(1) <= bound * np.maximum(top, 0 if potential else 1)).all()


@pytest.mark.parametrize("N,bound", [(256, 4.7e-15), (512, 9.4e-15), (2048, 3.1e-14)])
def test_fp64_states_of_a_few_steps(q, N, bound):  # noqa: F811
    """Final states of four steps, no further from 64-bit arithmetic than a transform through one N-point FFT leaves
    them (bound: its largest error over six seeds of such media).  The plans' running sum over 2/R of the spectrum is
    what sets the error here: radix 4 at N = 512 left 2.5e-14."""
    from paper_2107_06147_gb300 import inputs
    w = inputs.small_parity(N=N, n_traj=24, seed=2)
    w.grid.L, w.grid.dt = N * (5.0 / 256 if N <= 256 else 5.0 / 512), 0.001
    w.inits = [inputs.InitSpec("gauss", 0.8, 1, 0, 0), inputs.InitSpec("coulomb", 0.0, 1, 0, 0),
               inputs.InitSpec("coulomb", 0.0, 2, 0, 0), inputs.InitSpec("gauss", 0.8, 2, 1, 0)]
    w.init_idx = (np.arange(24) % 4).astype(np.int32)
    Tf = 0.42 * (0.6 / (0.6 + 3.5 * 0.1973269804 * 0.001)) ** (1 / 3)
    w.media = [inputs.MediumSpec(0.42, 0.6, Tf, k, g) for k in (4.0, 5.0, 6.0) for g in (-2.0, 0.0)]
    w.medium_idx = (np.arange(24) // 4).astype(np.int32)
    w.seeds = np.full(24, 117390, np.uint64)   # (a first threshold of 7e-7: no jump)
    ref, uref = run_oracle(w, use_rmin=0)
    obs, u = run_gpu(q, w, q.FP64, use_rmin=0)
    assert (ref["n_jumps"] == 0).all() and (obs["n_steps_exec"] == 4).all()
    assert np.linalg.norm(u - uref) <= bound * np.linalg.norm(uref), np.linalg.norm(u - uref) / np.linalg.norm(uref)


def _pulsed(T, dt, tau0):
    """A table with the temperatures T at the steps, constant around each step's time."""
    t = tau0 + np.arange(len(T)) * dt * 0.1973269804
    d = 0.3 * dt * 0.1973269804
    tau = np.stack([t - d, t + d], 1).ravel()
    tau[0] = tau0
    return tau, np.repeat(T, 2)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("N", [256, 2048])
def test_temperature_that_changes_within_a_step(q, N, precision):  # noqa: F811
    """The end-of-step norm is taken before the merged half-steps of two temperatures are applied; its weight has to
    hold for any change of T over a step, not only for the 1e-4 of a Bjorken medium: a rise and a fall by 2.5 within
    the first steps, on states whose exponents reach 5 a step."""
    import torch
    import oracle as o
    n, dt, kappa = 400, 0.02, 150.0
    tau, T = _pulsed(np.array([0.2, 0.5] + 8 * [0.2] + [0.5, 0.2, 0.2]), dt, 0.6)
    g = o.Grid(N=N, L=20.0, dt=dt, use_rmin=0)
    idx = (np.arange(n) % 2).astype(np.int32)
    seeds = np.arange(n, dtype=np.uint64)
    states = [("gauss", 2.0, 1, 0, 0), ("gauss", 3.0, 2, 1, 0)]
    ref, _, uref = o.run_batch(g, [o.init_spec(*s) for s in states], idx,
                               [o.table_medium(tau, T, Tf=0.15, kappa_hat=kappa, gamma_hat=-1.0)],
                               np.zeros(n, np.int32), seeds, want_states=True)
    assert (ref["n_steps_exec"] >= 12).all() and (ref["n_jumps"] > 0).mean() > 0.9
    e = q.Engine(q.Config(N=N, L=20.0, dt=dt, precision=precision, use_rmin=0, save_states=1))
    e.set_profiles(tau, T)
    e.init([q.init_spec(*s) for s in states], n, idx)
    e.evolve([q.table_medium(0, len(tau), 0.15, kappa, -1.0)], seeds, np.zeros(n, np.int32))
    obs, u = e.observables(), e.states()
    torch.cuda.synchronize()
    e.close()
    if precision == 0:
        check_fp64(q, obs, ref, u, uref)
    else:
        check_fp32(q, obs, ref, u, uref, min_same=0.98)


@pytest.mark.parametrize("N", [128, 512, 2048, 8192])
def test_fp32_exponents_beyond_single_precision(q, N):  # noqa: F811
    """A wide state on a long grid, kappa_hat 6 and 60: exponents to -11 and -109 and phases to -6 a step at the
    largest r.  The seed's first threshold (6.9e-7) is below every norm, so nothing jumps."""
    from paper_2107_06147_gb300 import inputs
    w = inputs.small_parity(N=N, n_traj=4, seed=1)
    w.grid.L, w.grid.dt = 200.0, 0.001
    w.inits = [inputs.InitSpec("gauss", 30.0, 1, 0, 0), inputs.InitSpec("gauss", 60.0, 2, 1, 0)]
    w.media = [inputs.MediumSpec(0.45, 0.6, 0.4495, 6.0, -3.5), inputs.MediumSpec(0.45, 0.6, 0.4495, 60.0, -3.5)]
    w.init_idx, w.medium_idx = np.array([0, 1, 0, 1], np.int32), np.array([0, 0, 1, 1], np.int32)
    w.seeds = np.full(4, 117390, np.uint64)
    ref, uref = run_oracle(w, use_rmin=0)
    obs, u = run_gpu(q, w, q.FP32, use_rmin=0)
    assert (ref["n_jumps"] == 0).all() and (obs["n_jumps"] == 0).all() and (ref["n_steps_exec"] == 11).all()
    bound = fp32_bound(N, ref["n_steps_exec"])
    du = np.linalg.norm(u - uref, axis=1) / np.linalg.norm(uref, axis=1)
    assert (du <= bound).all(), du / bound
    assert (np.abs(obs["norm2"] / ref["norm2"] - 1) <= 2 * bound).all(), obs["norm2"] / ref["norm2"] - 1


@pytest.mark.parametrize("Tf", [0.399, 0.39999])
@pytest.mark.parametrize("gamma", [0.0, -1.0])
def test_fp32_exponent_that_overflows_is_reported(q, gamma, Tf):  # noqa: F811
    """kappa_hat = 1e300 passes the host's checks and its coefficient is infinite in FP32: 0 x inf at r = 0 is not a
    number and is flagged, in media of one step and more, with jumps capped as well (no renormalisation of a zero
    state then)."""
    import torch
    e = q.Engine(q.Config(N=512, L=5.0, dt=0.001, precision=q.FP32, use_rmin=0, max_jumps=0))
    e.init([q.init_spec("gauss", 0.3, 1, 0, 0)], 2)
    e.evolve([q.medium(0.4, 0.6, Tf, 1e300, gamma)], np.arange(2, dtype=np.uint64))
    o = e.observables(check_finite=False)
    with pytest.raises(q.QtrajError) as ei:
        e.observables()
    torch.cuda.synchronize()
    e.close()
    assert ei.value.status == 5 and (o["flags"] & q.F_NONFINITE).all(), o["flags"]


def test_repeated_evolves_do_not_wait_for_the_first(q):  # noqa: F811
    """Three evolves queued on one stream: the third call prepares and returns while the first one's kernel runs (its
    descriptors may not wait for the second upload, which is queued behind that kernel)."""
    import torch
    n = 20000
    e = q.Engine(q.Config(N=1024, L=10.0, dt=0.001, precision=q.FP32, use_rmin=0))
    e.init([q.init_spec("gauss", 0.2, 1, 0, 0)], n)
    seeds = np.arange(n, dtype=np.uint64)
    long_, short = [q.medium(0.5, 0.6, 0.38, 3.0, -1.0)], [q.medium(0.5, 0.6, 0.499, 3.0, -1.0)]
    for _ in range(3):
        e.evolve(short, seeds)
    torch.cuda.synchronize()
    first = torch.cuda.Event()
    e.evolve(long_, seeds)
    first.record()
    e.evolve(short, seeds)
    e.evolve(short, seeds)
    running = not first.query()
    a = e.observables()
    torch.cuda.synchronize()
    e.evolve(short, seeds)
    b = e.observables()
    torch.cuda.synchronize()
    e.close()
    assert running
    assert np.array_equal(a["jump_digest"], b["jump_digest"]) and np.array_equal(a["norm2"], b["norm2"])


@pytest.mark.parametrize("N,variant", [(2048, 2), (4096, 3)])
def test_vacuum_evolution_under_the_radix_8_variants(q, N, variant):  # noqa: F811
    import oracle as o
    from paper_2107_06147_gb300 import inputs
    w = inputs.small_parity(N=N, n_traj=4, seed=35)
    for m in w.media:
        m.Tf = 0.99 * m.T0
    g, inits, media = oracle_inputs(w)
    g.t_vac, g.use_rmin = 0.05, 0
    ref, _, uref = o.run_batch(g, inits, w.init_idx, media, w.medium_idx, w.seeds, want_states=True)
    obs, u = run_gpu(q, w, q.FP32, t_vacuum=0.05, variant=variant, use_rmin=0)
    check_fp32(q, obs, ref, u, uref, min_same=0.75)


@pytest.mark.parametrize("N", [16, 128, 512, 2048, 4096, 8192])
def test_ksu_fp64_plans(q, N):  # noqa: F811
    """The FP64 KSU kernel on the plans that test_gpu_ksu leaves out, 1e-10 as there."""
    import oracle as o
    from oracle import eigen
    import torch
    g = o.Grid(N=N, L=12.0, dt=0.001, potential=1, use_rmin=0)
    e = q.Engine(q.Config(N=N, L=12.0, dt=0.001, precision=q.FP64, potential=1, save_states=1))
    states, T = [("gauss", 0.3, 1, 0, 0), ("gauss", 0.5, 2, 1, 0)], (0.4, 0.6, 0.396)
    g.basis = eigen.numerical_basis(g) if N <= 512 else e.basis()   # (the dense eigensolver of larger grids takes minutes)
    idx = np.arange(2, dtype=np.int32)
    ref, _, uref = o.run_batch(g, [o.init_spec(*s) for s in states], idx, [o.medium(*T, 0.0, 0.0)], np.zeros(2, np.int32),
                               np.arange(2, dtype=np.uint64), want_states=True)
    e.init([q.init_spec(*s) for s in states], 2, idx)
    e.evolve([q.medium(*T, 0.0, 0.0)], np.arange(2, dtype=np.uint64), np.zeros(2, np.int32))
    obs, u = e.observables(), e.states()
    torch.cuda.synchronize()
    e.close()
    assert (ref["n_steps_exec"] > 10).all() and np.array_equal(obs["n_steps_exec"], ref["n_steps_exec"])
    assert (np.linalg.norm(u - uref, axis=1) <= 1e-10 * np.linalg.norm(uref, axis=1)).all()
    assert (np.abs(obs["norm2"] / ref["norm2"] - 1) <= 1e-10).all()
    assert (np.abs(obs["surv"] - ref["surv"]).max(1) <= 1e-10 * np.maximum(1, ref["surv"].max(1))).all()
