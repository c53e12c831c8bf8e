"""pa_run_steps by the graphs of its steps: the same run as single steps when
checkpoints, adaptive steps, loaded populations and captures come between, in lockstep
with the oracle, and without waiting for the device."""
from __future__ import annotations

import time

import numpy as np
import pytest

from lockstep import compare_obs, compare_state, configs
from oracle import oracle as O

pytestmark = pytest.mark.gpu

# every resampling rule, bytes, and replicas with many copies (k_spread)
SPECS = [dict(dim=2, L=8, layout=1, R0=300, resample=0), dict(dim=2, L=16, layout=0, R0=200, resample=1),
         dict(dim=3, L=4, layout=1, model=1, coupling_seed=3, R0=200, resample=2),
         dict(dim=2, L=64, layout=1, R0=60, resample=2), dict(dim=2, L=16, layout=1, R0=300, beta_max=60.0)]
LONG = 300  # steps of a call that builds the graph


@pytest.fixture(scope="module")
def P():
    from paper_2006_00561_gb300 import build as B
    B.build()
    from paper_2006_00561_gb300 import pa
    return pa


def config(P, **kw):
    kw = dict(dict(K=600, theta=1, beta_max=1.0, seed=21), **kw)
    return P.make_config(**kw)


def same(P, a, b):
    sa, sb = a.state(), b.state()
    assert sa["status_bits"] == 0 and sa == sb
    for what in (P.DUMP_SPINS_RAW, P.DUMP_EBIN, P.DUMP_MAG, P.DUMP_HIST, P.DUMP_COUNTS, P.DUMP_OFFSETS,
                 P.DUMP_TAB_N, P.DUMP_TAB_F):
        assert np.array_equal(a.dump(what), b.dump(what)), what
    assert a.history(0, sa["step"] + 1) == b.history(0, sb["step"] + 1)


def singly(run, n):
    for _ in range(n):
        run.step()


by_spec = pytest.mark.parametrize("spec", SPECS, ids=lambda s: f"{s['dim']}d L={s['L']} R={s['R0']}")


@by_spec
@pytest.mark.parametrize("n", [1, 5, 7, 8, 9, 16, 17, 50])
def test_calls_of_any_length_without_waiting(P, spec, n):
    """From single launches over to graphs, of eight steps and of one."""
    a, b = P.Run(config(P, **spec)), P.Run(config(P, **spec))
    for _ in range(-(-150 // n)):
        a.run_steps(n)
        singly(b, n)
    same(P, a, b)


@by_spec
def test_restore_then_replay(P, spec):
    a, b = P.Run(config(P, **spec)), P.Run(config(P, **spec))
    a.run_steps(100)
    singly(b, 100)
    blob = b.checkpoint()
    a.run_steps(LONG)
    a.restore(blob)
    a.run_steps(33)
    singly(b, 33)
    same(P, a, b)


@by_spec
def test_adaptive_steps_and_loads_between_replays(P, spec):
    """Moved steps (their own weight tables), a lone resample and a loaded population
    between replays of the graph that was captured before them."""
    a, b = P.Run(config(P, **spec)), P.Run(config(P, **spec))
    a.run_steps(LONG)
    singly(b, LONG)
    for k in range(3):
        for run in (a, b):
            beta = run.observables()["beta"]
            run.resample_to(beta + (0.4 + 0.3 * k) / 600)
            run.sweep(1)
        a.run_steps(17)
        singly(b, 17)
    for run in (a, b):
        spins = run.spins()
        run.load(P.DUMP_SPINS, np.ascontiguousarray(spins), spins.shape[0])
        run.resample()
        run.sweep(2)
    a.run_steps(25)
    singly(b, 25)
    same(P, a, b)


@pytest.mark.parametrize("n", [2, 9, 40])
def test_runs_of_steps_in_lockstep_with_the_oracle(P, n):
    """Calls of several steps, whose observables share a launch with the reweight."""
    for spec in SPECS[:4]:
        ocfg, gcfg = configs(P, K=120, theta=1, beta_max=1.0, seed=22, **spec)
        orun, run = O.Run(ocfg), P.Run(gcfg)
        want = [orun.observables()]
        for i in range(1, 2 * n + 1):
            assert orun.step() == 0
            want.append(orun.observables())
            if i % n == 0:
                run.run_steps(n)
                compare_state(P, run, orun, i)
        for h, w in zip(run.history(0, 2 * n + 1), want):
            compare_obs(h, w)


def test_a_captured_call(P):
    """Under the caller's capture the steps are enqueued kernel by kernel."""
    import torch
    stream = torch.cuda.Stream()
    spec = SPECS[0]
    a, b = P.Run(config(P, **spec), stream=stream), P.Run(config(P, **spec))
    a.run_steps(LONG)
    singly(b, LONG)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
        a.run_steps(100)
    with torch.cuda.stream(stream):
        graph.replay()
        graph.replay()
    torch.cuda.synchronize()
    singly(b, 200)
    same(P, a, b)


@pytest.mark.parametrize("calls", [(200,), (1,) * 200, (20,) * 10], ids=["one call", "of one", "of twenty"])
@pytest.mark.parametrize("rule", [0, 2])
def test_the_call_does_not_wait_for_the_device(P, rule, calls):
    """200 steps of some 1.6 ms: far more kernels than the launch queue holds."""
    import torch
    run = P.Run(config(P, dim=2, L=64, R0=1 << 16, theta=10, resample=rule))
    run.run_steps(1)
    assert run.status() == 0
    t0 = time.perf_counter()
    for n in calls:
        run.run_steps(n)
    host = time.perf_counter() - t0
    torch.cuda.synchronize()
    total = time.perf_counter() - t0
    assert run.status() == 0 and host < 0.1 * total, (host, total)
