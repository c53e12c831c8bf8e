"""The autotuner tries the shapes that differ for a class's kernel, once each, and
does not take a choice that was saved when the shapes meant something else."""
from __future__ import annotations

import json

import pytest

pytest.importorskip("torch")

from paper_2006_00561_gb300 import autotune  # noqa: E402
from test_autotune_host import FakeBatch, cls, fake_cuda  # noqa: E402, F401


@pytest.mark.parametrize("layout,L", [(0, 16), (0, 64), (1, 16)])
def test_two_forms_of_the_sliced_kernel(fake_cuda, layout, L):  # noqa: F811
    c = dict(cls(2, L, 100_000), layout=layout, kernel="sliced")
    b = FakeBatch([c], {(0, 2): 1.0, (0, 4): 2.0, (0, 8): 1.5})
    out = autotune.tune(b, steps_left=100, cache_path=None)
    assert out["shapes"] == {0: (8, 0)} and out["steps_used"] == 2


def test_register_kernels_search_slots_per_claim(fake_cuda):  # noqa: F811
    c = dict(cls(2, 64, 100_000, warps=12), kernel="register")
    b = FakeBatch([c], {(0, 12): 1.0}, {(0, 8): -0.5})
    out = autotune.tune(b, steps_left=100, cache_path=None)
    assert out["shapes"] == {0: (12, 8)} and out["steps_used"] == len(autotune.CHUNKS)


def test_a_choice_saved_for_the_earlier_kernel_is_measured_again(fake_cuda, tmp_path):  # noqa: F811
    path = tmp_path / "tune.json"
    path.write_text(json.dumps({"FakeGPU|layout1|d3|L8|m1|slots4194304": [8, 0]}))
    b = FakeBatch([cls(3, 8, 3_000_000)], {(0, 2): 9.0, (0, 4): 7.0, (0, 8): 8.0})
    out = autotune.tune(b, steps_left=100, cache_path=str(path))
    assert out["shapes"] == {0: (4, 0)} and out["steps_used"] == 3


@pytest.mark.gpu
def test_classes_name_their_kernel():
    from paper_2006_00561_gb300 import build as B
    B.build()
    from paper_2006_00561_gb300 import pa as P
    runs = [P.Run(P.make_config(dim=d, L=L, layout=layout, R0=40, K=4, theta=1))
            for d, L, layout in ((2, 64, 1), (2, 64, 0), (2, 128, 1), (2, 16, 1), (3, 8, 0))]
    batch = P.Batch(runs)
    kernels = {(c["dim"], c["L"], c["layout"]): c["kernel"] for c in batch.classes()}
    assert kernels == {(2, 64, 1): "register", (2, 64, 0): "sliced", (2, 128, 1): "register",
                       (2, 16, 1): "sliced", (3, 8, 0): "sliced"}
    out = autotune.tune(batch, steps_left=4, cache_path=None)
    assert out["steps_used"] == 4 and batch.sync() == 0
    batch.close()
