"""Inputs at the ends of their ranges: states decayed below FP32's products, temperatures that drop within a step,
exponents beyond FP32's, and repeated calls that may not wait for each other."""
import numpy as np
import pytest

from test_gpu_parity import check_fp32, check_fp64, fp32_bound, oracle_inputs, q, run_gpu, run_oracle  # noqa: F401

pytestmark = pytest.mark.gpu


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
