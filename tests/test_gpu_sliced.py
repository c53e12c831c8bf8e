"""The replica-sliced sweep in all of its forms, every lattice and layout:
populations around a chunk of replicas, populations on both sides of the
line between four lanes per group and one, and batched classes in every block
shape.  Bit for bit against the oracle."""
from __future__ import annotations

import pytest

from lockstep import compare_state, configs, run_lockstep
from oracle import oracle as O

pytestmark = pytest.mark.gpu

FOUR_BELOW = 2432  # warps of the one-lane form from which it is taken
LATTICES = [(2, 4), (2, 8), (2, 16), (2, 32), (2, 64), (2, 128),
            (3, 2), (3, 4), (3, 6), (3, 8), (3, 10), (3, 12), (3, 16)]


@pytest.fixture(scope="module")
def P():
    from paper_2006_00561_gb300 import build as B
    B.build()
    from paper_2006_00561_gb300 import pa
    return pa


def spec(dim, L, layout, model, **kw):
    return dict(dim=dim, L=L, layout=layout, model=model, beta_max=1.0 + model, seed=7 * L + dim,
                coupling_seed=L if model else 0, instance_id=L + model, **kw)


@pytest.mark.parametrize("model", [0, 1])
@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("dim,L", LATTICES)
def test_small_populations(P, dim, L, layout, model):
    for R0 in ((1, 33) if L ** dim > 2000 else (1, 31, 32, 33, 97)):
        run_lockstep(P, steps=2, R0=R0, K=30, theta=2, **spec(dim, L, layout, model))


@pytest.mark.parametrize("side", [-1, 1])
@pytest.mark.parametrize("dim,L,layout,model", [(2, 16, 0, 0), (2, 32, 1, 1), (2, 64, 0, 1),
                                                (2, 128, 0, 0), (3, 8, 0, 1), (3, 10, 1, 0),
                                                (3, 10, 0, 1), (3, 16, 1, 1)])
def test_populations_around_the_line_between_the_forms(P, dim, L, layout, model, side):
    per_chunk = (L ** dim // 8 + 31) // 32
    chunks = -(-FOUR_BELOW // per_chunk)  # the fewest that take one lane per group
    R0 = 32 * (chunks - 1) + (1 if side > 0 else 0)
    run_lockstep(P, steps=1, R0=R0, K=20, theta=1, **spec(dim, L, layout, model))


@pytest.mark.parametrize("dim,L,layout,model,R0",
                         [(2, 16, 0, 0, 4801), (2, 16, 1, 1, 9999), (2, 32, 0, 0, 1999),
                          (2, 32, 1, 0, 4701), (3, 6, 1, 1, 4099), (3, 6, 0, 0, 7900),
                          (3, 8, 1, 1, 2001), (3, 10, 0, 1, 2003), (3, 10, 1, 1, 4050),
                          (3, 12, 1, 0, 1601), (2, 64, 0, 1, 1700)])
def test_chunks_of_16_and_32_replicas(P, dim, L, layout, model, R0):
    """Smaller populations take chunks of eight (test_small_populations)."""
    run_lockstep(P, steps=1, R0=R0, K=20, theta=1, **spec(dim, L, layout, model))


@pytest.mark.parametrize("warps", [2, 4, 8])
def test_batched_classes_in_every_shape(P, warps):
    mix = [(2, 8, 1, 0, 70), (2, 16, 0, 1, 64), (2, 64, 0, 0, 33), (2, 128, 0, 1, 5), (3, 6, 1, 1, 200),
           (3, 6, 1, 1, 31), (3, 10, 1, 1, 65), (3, 10, 0, 0, 40), (3, 12, 1, 1, 34), (3, 16, 1, 0, 33)]
    runs, oracles = [], []
    for i, (dim, L, layout, model, R0) in enumerate(mix):
        s = spec(dim, L, layout, model, R0=R0, K=20, theta=2)
        s["seed"] += i
        ocfg, gcfg = configs(P, **s)
        oracles.append(O.Run(ocfg))
        runs.append(P.Run(gcfg))
    batch = P.Batch(runs)
    for c in range(len(batch.classes())):
        batch.set_shape(c, warps, 0)
        assert batch.classes()[c]["warps"] == warps
    for i in (1, 2):
        batch.step()
        assert batch.sync() == 0
        for r, o in zip(runs, oracles):
            assert o.step() == 0
            compare_state(P, r, o, i)
    batch.close()


@pytest.mark.parametrize("L,model,R0", [(64, 0, 151), (64, 0, 153), (64, 0, 16 * 152 + 1),
                                        (64, 1, 12 * 152 + 1), (128, 0, 151), (128, 0, 8 * 152 + 3),
                                        (128, 0, 12 * 152 - 60), (128, 1, 8 * 152 + 1)])
def test_register_kernels_around_a_round(P, L, model, R0):
    """Replicas dealt to the SMs one by one, in one round or a little more, and
    both block sizes of the L = 128 ferromagnet."""
    run_lockstep(P, steps=1, R0=R0, K=20, theta=1, **spec(2, L, 1, model))
