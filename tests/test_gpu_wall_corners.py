"""Particles in the corners of a box with walls on every side, for both lattices
and box sides that are no multiples of the 32x4x2 bricks: the rows of those
bricks start and end at a wall (and, ragged, inside the brick).  One step
against the oracle, with the tolerances of tests/test_gpu_parity.py.

"corners" has a few near bricks; "filled" lets 7680 be expected, some 50 per SM,
which the near sweep's other form takes."""
import itertools

import numpy as np
import pytest

from tests import _helpers as H

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts
    pytest.skip("no CUDA device", allow_module_level=True)

from tests.test_gpu_parity import _compare_step, W, pkg  # noqa: E402,F401


def workload(W, box):
    wl = W.empty_box(8, "f32", (0, 0, 0))
    if box == "corners":
        n, per_axis = (33, 21, 19), (2, 2, 2)
    else:
        n, per_axis = (97, 58, 65), (8, 4, 5)
    wl.update(nx=n[0], ny=n[1], nz=n[2], tau=0.8)
    axes = [np.linspace(2.3, m - 1 - 2.3, k) for m, k in zip(n, per_axis)]
    wl["particles"] = [W._particle([[0.7, 0.1, -0.2], [-0.7, -0.1, 0.2]], [2.5, 2.5], c, q=(0.8, 0.3, -0.4, 0.33),
                                   v=(0.01, -0.02, 0.015), w=(0.002, -0.001, 0.003), density=1.2, fixed=1)
                       for c in itertools.product(*axes)]
    return H.fixed_mass(wl)


@pytest.mark.parametrize("box", ["corners", "filled"])
@pytest.mark.parametrize("storage,Q", [("f32", 15), ("f32", 19), ("f64", 15), ("f16", 15)])
def test_one_step(pkg, oracle_mod, W, box, storage, Q):  # noqa: F811
    _compare_step(pkg, oracle_mod, workload(W, box), storage, Q=Q)
