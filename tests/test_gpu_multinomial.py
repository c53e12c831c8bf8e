"""Multinomial draws over more tiles than the GPU holds CTAs, and around the
1024 tiles up to which a search begins on every tile's end: against the oracle."""
from __future__ import annotations

import pytest

from lockstep import run_lockstep

pytestmark = pytest.mark.gpu

TILE, TOP = 2048, 1024


@pytest.fixture(scope="module")
def P():
    from paper_2006_00561_gb300 import build as B
    B.build()
    from paper_2006_00561_gb300 import pa
    return pa


@pytest.mark.parametrize("R0", [TOP * TILE, TOP * TILE + 30_001, 2 * TOP * TILE + 1],
                         ids=["spans of one tile", "of two", "of three"])
def test_draws_over_thousands_of_tiles(P, R0):
    run_lockstep(P, steps=2, dim=2, L=4, layout=1, R0=R0, K=8, theta=1, beta_max=1.0, seed=R0 & 0xffff,
                 resample=2)
