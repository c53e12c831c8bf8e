"""A step's kernels as a chain of dependent launches, single and from the CUDA
graph of several steps that a long pa_run_steps call builds, with every
resampling rule and sweep kernel: the same run, step for step."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SPECS = [dict(dim=2, L=8, layout=1, R0=300, resample=0), dict(dim=2, L=16, layout=0, R0=500, resample=1),
         dict(dim=3, L=6, layout=1, model=1, coupling_seed=3, R0=200, resample=2),
         dict(dim=2, L=64, layout=1, R0=100, resample=0), dict(dim=2, L=128, layout=1, R0=40, resample=1)]


@pytest.fixture(scope="module")
def P():
    from paper_2006_00561_gb300 import build as B
    B.build()
    from paper_2006_00561_gb300 import pa
    return pa


@pytest.mark.parametrize("spec", SPECS, ids=lambda s: f"{s['dim']}d L={s['L']} rule {s['resample']}")
@pytest.mark.parametrize("calls", [(256, 7, 30, 8), (255, 46)])
def test_long_calls_equal_single_steps(P, spec, calls):
    """256 steps build the graph, 7 run without it, 30 and 8 with it."""
    cfg = P.make_config(K=400, theta=1, beta_max=1.0, seed=12, **spec)
    a, b = P.Run(cfg), P.Run(cfg)
    for n in calls:
        a.run_steps(n)
        for _ in range(n):
            b.step()
        sa, sb = a.state(), b.state()
        assert sa["status_bits"] == 0 and sa == sb
        for what in (P.DUMP_SPINS_RAW, P.DUMP_EBIN, P.DUMP_MAG, P.DUMP_HIST, P.DUMP_COUNTS,
                     P.DUMP_OFFSETS):
            assert np.array_equal(a.dump(what), b.dump(what)), what
    done = sum(calls)
    assert a.history(0, done + 1) == b.history(0, done + 1)


def test_a_lone_resample_keeps_the_histogram(P):
    """Only the resample inside a whole step clears the histogram."""
    cfg = P.make_config(dim=2, L=8, layout=1, R0=500, K=20, theta=1, seed=5)
    run = P.Run(cfg)
    run.step()
    hist = run.dump(P.DUMP_HIST)
    run.resample()
    assert np.array_equal(run.dump(P.DUMP_HIST), hist) and hist.sum() == run.state()["R_prev"]
    run.sweep(1)
    assert run.dump(P.DUMP_HIST).sum() == run.state()["R"] and run.status() == 0


def test_stepping_past_K_after_a_long_call(P):
    run = P.Run(P.make_config(dim=2, L=4, layout=1, R0=50, K=256, theta=1, seed=6))
    run.run_steps(256)
    assert run.status() == 0
    run.run_steps(3)
    assert run.status() == -8
