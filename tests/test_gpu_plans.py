"""Every plan of the sine transform (radices, one or two middle passes, slots of 4 to 32 values, fused and
plain kernels, the launch variants and their traced twins) against the CPU oracle over a short medium, with the
tolerances of test_gpu_parity; and the FP32 potential factor outside its series' range."""
import numpy as np
import pytest

from test_gpu_parity import check_fp32, check_fp64, fp32_bound, q, run_gpu, run_oracle  # noqa: F401

pytestmark = pytest.mark.gpu


def _short(N, n_traj, seed):
    from paper_2107_06147_gb300 import inputs
    w = inputs.small_parity(N=N, n_traj=n_traj, seed=seed)
    for m in w.media:
        m.Tf = m.T0 * (0.97 if N <= 1024 else 0.99)
    return w


@pytest.mark.parametrize("N", [16, 32, 64, 128, 256, 512, 1024, 2048, 4096, 8192])
def test_fp64_plans(q, N):  # noqa: F811
    w = _short(N, 6, N + 5)
    ref, uref = run_oracle(w, use_rmin=0)
    obs, u = run_gpu(q, w, q.FP64, use_rmin=0)
    check_fp64(q, obs, ref, u, uref)


@pytest.mark.parametrize("N", [32, 128, 512, 2048, 4096, 8192, 16384])
def test_plain_plans(q, N):  # noqa: F811
    w = _short(N, 5, N + 6)
    ref, uref = run_oracle(w, use_rmin=0)
    obs, u = run_gpu(q, w, q.FP64, form=q.PLAIN, use_rmin=0)
    check_fp64(q, obs, ref, u, uref)


@pytest.mark.parametrize("N,variant", [(16, 0), (32, 0), (128, 0), (256, 0), (512, 0), (1024, 0), (2048, 0), (2048, 1),
                                       (2048, 2), (2048, 3), (4096, 1), (4096, 2), (4096, 3)])
def test_fp32_plans(q, N, variant):  # noqa: F811
    w = _short(N, 6, N + 7)
    ref, uref = run_oracle(w, use_rmin=0)
    obs, u = run_gpu(q, w, q.FP32, use_rmin=0, variant=variant)
    check_fp32(q, obs, ref, u, uref, min_same=0.8)


@pytest.mark.parametrize("N,variant", [(2048, 0), (2048, 3), (4096, 2)])
def test_traced_twin_gives_the_same_records(q, N, variant):  # noqa: F811
    """The traced kernel runs the context's own plan: its rows end on the record's norm, and the records are the
    untraced ones."""
    import torch
    w = _short(N, 4, 3)
    e = q.Engine(q.Config(N=N, L=w.grid.L, dt=w.grid.dt, precision=q.FP32, use_rmin=0, variant=variant))
    e.init([q.init_spec(s.kind, s.width, s.n, s.l, s.color) for s in w.inits], 4, w.init_idx)
    media = [q.medium(m.T0, m.tau0, m.Tf, m.kappa_hat, m.gamma_hat) for m in w.media]
    e.evolve(media, w.seeds, w.medium_idx)
    a = e.observables()
    e.set_trace(every=10, n_traced=2, max_records=64)
    e.evolve(media, w.seeds, w.medium_idx)
    b = e.observables()
    rows = e.trace()
    torch.cuda.synchronize()
    e.close()
    assert np.array_equal(a["jump_digest"], b["jump_digest"])
    bound = fp32_bound(N, a["n_steps_exec"])
    assert (np.abs(a["norm2"] / b["norm2"] - 1) <= bound).all()
    for t in range(2):
        assert rows[t]["step"][-1] == b["n_steps_exec"][t]
        if b["last_jump_step"][t] != b["n_steps_exec"][t] - 1:   # (a row is written before its step's jump)
            assert abs(rows[t]["norm2"][-1] / b["norm2"][t] - 1) <= bound[t]


@pytest.mark.parametrize("N", [512, 2048])
def test_fp32_factor_beyond_its_series(q, N):  # noqa: F811
    """A wide state on a long grid: exponents to -20 and phases to -10 a step at the largest r, where the factor's
    arguments are reduced to the series' range; jumps are suppressed (max_jumps large, thresholds met at random)."""
    w = _short(N, 6, 4)
    from paper_2107_06147_gb300 import inputs
    w.grid.L = 200.0
    w.inits = [inputs.InitSpec("gauss", 30.0, 1, 0, 0), inputs.InitSpec("gauss", 60.0, 2, 1, 0)]
    w.init_idx[:] = np.arange(6) % 2
    w.media = [inputs.MediumSpec(0.45, 0.6, 0.4495, 6.0, -3.5), inputs.MediumSpec(0.45, 0.6, 0.4495, 0.5, -3.5)]
    w.medium_idx[:] = np.arange(6) // 2 % 2
    ref, uref = run_oracle(w, use_rmin=0)
    obs, u = run_gpu(q, w, q.FP32, use_rmin=0)
    same = obs["jump_digest"] == ref["jump_digest"]
    assert same.mean() >= 0.5
    du = np.linalg.norm(u[same] - uref[same], axis=1) / np.linalg.norm(uref[same], axis=1)
    assert (du <= fp32_bound(N, ref["n_steps_exec"][same])).all(), du


@pytest.mark.parametrize("gamma", [-1e4, -1e7, -1e11])
def test_fp32_large_phases_conserve_the_norm(q, gamma):  # noqa: F811
    """kappa_hat = 0 is unitary whatever the phase: phases of 1 to 10^7 a step, through the reduced series and, above
    10^5, the library's."""
    import torch
    e = q.Engine(q.Config(N=64, L=2.5, dt=0.001, precision=q.FP32, use_rmin=0, max_jumps=0))
    e.init([q.init_spec("gauss", 0.3, 1, 0, 0), q.init_spec("gauss", 0.3, 2, 1, 0)], 2)
    e.evolve([q.medium(0.4, 0.6, 0.399, 0.0, gamma)], np.array([11, 12], np.uint64))
    o = e.observables()
    torch.cuda.synchronize()
    e.close()
    assert (o["n_steps_exec"] > 10).all()
    assert (np.abs(o["norm2"] - 1) <= fp32_bound(64, o["n_steps_exec"])).all(), o["norm2"]


def test_static_entry_takes_no_flags_of_an_earlier_call(q):  # noqa: F811
    """A KSU call of qtraj_evolve_static (no groups, use_rmin on by default) after an OQS call whose groups published
    their no-jump records in the shared scratch: the records are the KSU evolution's, as through a workspace."""
    import ctypes as C
    import torch
    spec, med = q.init_spec("gauss", 0.8, 1, 0, 0), q.medium(0.425, 0.6, 0.4, 0.5, 0.0)
    seeds = np.arange(4, dtype=np.uint64)

    def static(e):
        out = torch.zeros(4 * q.OBS_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
        st = e.lib.qtraj_evolve_static(e.ctx, 4, (q.InitSpec * 1)(spec), 1, None, (q.Medium * 1)(med), 1, None,
                                       seeds.ctypes.data_as(C.POINTER(C.c_uint64)), C.c_void_p(out.data_ptr()),
                                       C.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert st == 0, e.lib.qtraj_last_error(e.ctx)
        return out.cpu().numpy().view(q.OBS_DTYPE)

    oqs = q.Engine(q.Config(N=64, L=5.0, dt=0.001, precision=q.FP64))
    static(oqs)
    ksu = q.Engine(q.Config(N=64, L=5.0, dt=0.001, precision=q.FP64, potential=1))
    a = static(ksu)
    ksu.init([spec], 4)
    ksu.evolve([med], seeds)
    b = ksu.observables()
    assert (a["n_steps_exec"] > 0).all() and np.array_equal(a["norm2"], b["norm2"]) and np.array_equal(a["surv"], b["surv"])
    oqs.close()
    ksu.close()
