"""The resample's tiles, their slices and the block-wide lookback at the sizes
where they change: populations around the edges, capacities on both sides of a
slice width, more tiles than one lookback window holds, and the allocation-free scan
on buffers that are not 16-byte aligned.  Bit for bit against the oracle."""
from __future__ import annotations

import math

import numpy as np
import pytest

from lockstep import compare_state, configs, run_lockstep
from oracle import oracle as O

pytestmark = pytest.mark.gpu

TILE, SPREAD = 2048, 608  # tiles that fill the GPU with one CTA each


@pytest.fixture(scope="module")
def P():
    from paper_2006_00561_gb300 import build as B
    B.build()
    from paper_2006_00561_gb300 import pa
    return pa


# a single replica under the Poisson rule dies out in the oracle too
@pytest.mark.parametrize("R0,rule", [(1, 0), (1, 2)] + [(R0, rule) for R0 in (31, 32, 33, 65, 2049)
                                                        for rule in (0, 1, 2)])
def test_populations_around_a_tile(P, R0, rule):
    run_lockstep(P, steps=4, dim=2, L=8, layout=1, R0=R0, K=8, theta=1, beta_max=0.4,
                 seed=500 + R0, resample=rule)


@pytest.mark.parametrize("tiles", [SPREAD // 64, SPREAD // 64 + 1, SPREAD // 2, SPREAD // 2 + 1])
def test_capacities_around_a_slice_width(P, tiles):
    """R0 fills the capacity but for the room its fluctuations need."""
    capacity = TILE * tiles
    R0 = capacity - 16 * math.isqrt(capacity)
    run_lockstep(P, steps=2, dim=2, L=4, layout=1, R0=R0, capacity=capacity, K=8, theta=1,
                 beta_max=1.0, seed=capacity & 0xffff)


def test_batch_of_small_and_large_runs_shares_one_slice_width(P):
    """Runs whose own slices are narrower than the batch's, of every rule."""
    specs = [dict(dim=2, L=4, layout=1, R0=R0, K=6, theta=1, beta_max=0.8, seed=40 + i, resample=rule)
             for i, (R0, rule) in enumerate(((7, 0), (300, 1), (9000, 2), (17000, 1), (70000, 0)))]
    runs, oracles = [], []
    for s in specs:
        ocfg, gcfg = configs(P, **s)
        oracles.append(O.Run(ocfg))
        runs.append(P.Run(gcfg))
    batch = P.Batch(runs)
    for i in range(1, 4):
        if i == 2:  # a plain step of every run in between, on its own slices
            for r in runs:
                r.step()
        else:
            batch.step()
            assert batch.sync() == 0
        for r, o in zip(runs, oracles):
            assert o.step() == 0
            compare_state(P, r, o, i)
    batch.close()


@pytest.mark.parametrize("shift", [0, 1, 2])
@pytest.mark.parametrize("R", [1, 5, 2047, 2048, 2049, 700_001])
def test_allocation_free_scan_at_any_alignment(P, R, shift):
    import torch
    bins = 513
    rng = np.random.default_rng(R + shift)
    ebin = rng.integers(0, bins, size=R, dtype=np.uint32)
    n = rng.integers(0, 3, size=bins, dtype=np.uint32)
    F = rng.integers(0, 1 << 32, size=bins, dtype=np.uint64).astype(np.uint32)

    def dev(a):  # `shift` words past an aligned address
        buf = torch.zeros(a.size + shift, dtype=torch.int32, device="cuda")
        buf[shift:] = torch.from_numpy(a.view(np.int32)).cuda()
        return buf

    d_e, d_n, d_F = dev(ebin), dev(n), dev(F)
    out = [torch.full((R + shift + 8,), -1, dtype=torch.int32, device="cuda") for _ in range(2)]
    total = torch.empty(1, dtype=torch.int32, device="cuda")
    at = 4 * shift
    P.pa_copy_counts_scan_noalloc(d_e.data_ptr() + at, R, d_n.data_ptr() + at, d_F.data_ptr() + at,
                                  bins, 77, 9, 3, out[0].data_ptr() + at, out[1].data_ptr() + at,
                                  total.data_ptr(), torch.cuda.current_stream().cuda_stream)
    counts, offsets = (t.cpu().numpy().view(np.uint32) for t in out)
    want = O.copy_counts(O.make_config(seed=77, instance_id=3), 9, ebin, n, F)
    assert np.array_equal(counts[shift:shift + R], want)
    scan = np.zeros_like(want)
    np.cumsum(want[:-1], out=scan[1:], dtype=np.uint32)
    assert np.array_equal(offsets[shift:shift + R], scan)
    assert int(total.cpu().numpy().view(np.uint32)[0]) == int(want.astype(np.int64).sum())
    for a in (counts, offsets):  # nothing outside the caller's range is written
        assert (a[:shift] == 0xffffffff).all() and (a[shift + R:] == 0xffffffff).all()


SKEWED = [dict(dim=2, L=32, layout=1, R0=3000, K=4, beta_max=2.0), dict(dim=2, L=16, layout=0, R0=5000, K=6),
          dict(dim=3, L=6, layout=1, model=1, coupling_seed=9, R0=2100, K=3, beta_max=3.0),
          dict(dim=2, L=64, layout=1, R0=700, K=40), dict(dim=2, L=4, layout=1, R0=9000, K=2, beta_max=3.0)]


@pytest.mark.parametrize("rule", [0, 1, 2])
@pytest.mark.parametrize("spec", SKEWED, ids=lambda s: f"{s['dim']}d L={s['L']}")
def test_beta_steps_that_leave_few_survivors(P, spec, rule):
    """Replicas with tens to thousands of copies, shared out to all CTAs."""
    run_lockstep(P, steps=2, theta=1, seed=31, resample=rule, **spec)


def test_batch_with_few_survivors(P):
    runs, oracles = [], []
    for i, s in enumerate(SKEWED + [dict(dim=2, L=16, layout=1, R0=300, K=50)]):
        ocfg, gcfg = configs(P, theta=1, seed=50 + i, resample=i % 3, **s)
        oracles.append(O.Run(ocfg))
        runs.append(P.Run(gcfg))
    batch = P.Batch(runs)
    for i in (1, 2):
        batch.step()
        assert batch.sync() == 0
        for r, o in zip(runs, oracles):
            assert o.step() == 0
            compare_state(P, r, o, i)
    batch.close()


@pytest.mark.parametrize("R0", [2047, 2048, 6145, 400_003])
def test_multinomial_draws_over_several_tiles(P, R0):
    run_lockstep(P, steps=2, dim=2, L=4, layout=1, R0=R0, K=8, theta=1, beta_max=1.0, seed=R0,
                 resample=2)
