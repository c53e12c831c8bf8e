"""Populations loaded in the device layout: only the bits of the lattice's sites
are spins, whatever else the row words of a lattice narrower than 32 hold."""
from __future__ import annotations

import numpy as np
import pytest

from lockstep import compare_state, configs
from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2006_00561_gb300 import build as B
    B.build()
    from paper_2006_00561_gb300 import pa
    return pa


@pytest.mark.parametrize("R0", [100, 40_000])  # chunks of 8 and 16 replicas, and of 32
@pytest.mark.parametrize("dim,L", [(2, 4), (2, 8), (2, 16), (3, 2), (3, 6), (3, 10), (3, 12)])
def test_bits_beyond_a_row_are_not_spins(P, dim, L, R0):
    spec = dict(dim=dim, L=L, model=dim - 2, layout=1, R0=R0, K=4, theta=1, seed=17)
    ocfg, gcfg = configs(P, **spec)
    orun, run = O.Run(ocfg), P.Run(gcfg)
    words = run.dump(P.DUMP_SPINS_RAW).view(np.uint32).reshape(R0, -1).copy()
    words[:, : L ** (dim - 1)] |= np.uint32((0xffffffff << L) & 0xffffffff)
    run.load(P.DUMP_SPINS_RAW, words, R0)
    compare_state(P, run, orun, 0)
    run.step()
    assert orun.step() == 0
    compare_state(P, run, orun, 1)
