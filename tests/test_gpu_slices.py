"""The resample's slices at the sizes where their width changes: capacities on
both sides of a change, for every width that a population or a batch can get.
Bit for bit against the oracle."""
from __future__ import annotations

import math

import pytest

from lockstep import compare_state, configs, run_lockstep
from oracle import oracle as O

pytestmark = pytest.mark.gpu

TILE, CTAS = 2048, 608  # replicas of a tile; CTAs that fill the GPU


def width_lg(stride: int, total: int, least: int) -> int:
    """log2 of the slices of a tile (resample_slices in pa_internal.cuh)."""
    target, lg = max(total // CTAS, least), 0
    while TILE >> (lg + 1) >= 32 and (TILE >> lg) * stride > target:
        lg += 1
    return lg


def stride_of(s: dict) -> int:
    N, rows = s["L"] ** s["dim"], s["L"] ** (s["dim"] - 1)
    return -(-(N if s["layout"] == 0 else 4 * rows * -(-s["L"] // 32)) // 16) * 16


@pytest.fixture(scope="module")
def P():
    from paper_2006_00561_gb300 import build as B
    B.build()
    from paper_2006_00561_gb300 import pa
    return pa


def first_capacity(lg: int) -> int:
    """The smallest capacity with slices of 2^-lg tiles, whatever a replica's bytes."""
    return CTAS * TILE >> lg


# width below and from the edge, and the copy rule; the widest that a replica's bytes
# allow (16 KB a slice at least) is the first of its lattice
EDGES = [(dict(dim=2, L=4, layout=1), 1, 0, 0), (dict(dim=2, L=4, layout=1), 1, 0, 2),
         (dict(dim=2, L=16, layout=1), 2, 1, 0), (dict(dim=3, L=4, layout=0), 3, 2, 1),
         (dict(dim=2, L=16, layout=0), 4, 3, 2), (dict(dim=3, L=8, layout=1), 5, 4, 0),
         (dict(dim=2, L=64, layout=1), 6, 5, 1)]


@pytest.mark.parametrize("spec,below,above,rule", EDGES, ids=lambda v: str(v) if isinstance(v, int) else
                         f"{v['dim']}d L={v['L']} layout {v['layout']}")
def test_capacities_on_both_sides_of_a_slice_width(P, spec, below, above, rule):
    stride, edge = stride_of(spec), first_capacity(above)
    for capacity, lg in ((edge - 1, below), (edge, above)):
        assert width_lg(stride, capacity * stride, 1 << 14) == lg
        run_lockstep(P, steps=1, R0=capacity - 8 * math.isqrt(capacity), capacity=capacity, K=20, theta=0,
                     beta_max=0.5, seed=capacity & 0xffff, resample=rule, model=spec["dim"] - 2, **spec)


def test_batch_of_runs_with_widths_of_their_own(P):
    """A batch of small and large replicas: its slices go by the bytes of all runs."""
    specs = [dict(dim=2, L=4, layout=1, R0=70_000), dict(dim=2, L=64, layout=1, R0=9000),
             dict(dim=2, L=16, layout=0, R0=20_000), dict(dim=2, L=128, layout=1, R0=600)]
    specs = [dict(s, K=20, theta=1, beta_max=0.5, seed=60 + i, resample=i % 3) for i, s in enumerate(specs)]
    runs, oracles = [], []
    for s in specs:
        ocfg, gcfg = configs(P, **s)
        oracles.append(O.Run(ocfg))
        runs.append(P.Run(gcfg))
    sizes = [(st["stride"], st["capacity"]) for st in (r.state() for r in runs)]
    total = sum(a * b for a, b in sizes)
    lgs = [width_lg(stride, total, 1 << 16) for stride, _ in sizes]
    assert len(set(lgs)) == len(lgs) and lgs != [width_lg(s, s * c, 1 << 14) for s, c in sizes]
    batch = P.Batch(runs)
    for i in range(1, 3):
        batch.step()
        assert batch.sync() == 0
        for r, o in zip(runs, oracles):
            assert o.step() == 0
            compare_state(P, r, o, i)
    batch.close()
