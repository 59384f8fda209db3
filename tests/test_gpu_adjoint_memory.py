"""The drag gradient from checkpoints against the one from every step's kept
data: J to the bit, each component to the spread of the FP32 atomics (1e-5 of the
largest, as in tests/test_gpu_adjoint.py), for runs whose last segment is whole
(T = 36, 100) and one to eight steps short; a ragged box."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts
    pytest.skip("no CUDA device", allow_module_level=True)

from tests.test_gpu_adjoint_modes import CP, K, pkg, scaled  # noqa: E402,F401


def engine(pkg, T, W, keep):  # noqa: F811
    from paper_2206_11634_gb300.adjoint import AdjointDrag
    c = CP.mean(axis=0)
    p = pkg.make_particle(CP - c, K, c, fixed=1, mass=1.0, inertia=np.eye(3))
    return AdjointDrag(33, 35, 31, particle=p, T=T, W=W, tau=0.8, force=(4e-6, 1e-6, 0.0), u0=(0.02, 0.0, 0.0),
                       keep_steps=keep)


@pytest.mark.parametrize("T,W", [(1, 1), (2, 1), (23, 9), (36, 10), (37, 37), (43, 10), (45, 5), (50, 50), (100, 30),
                                 (101, 20)])
def test_checkpoints_against_kept_steps(pkg, T, W):  # noqa: F811
    few, full = engine(pkg, T, W, False), engine(pkg, T, W, True)
    assert few.ws.numel() < full.ws.numel() or T < 30  # (fewer steps than that take less than their checkpoints)
    Ja, Jb = few.forward_np(CP, K), full.forward_np(CP, K)
    assert Ja == Jb != 0.0
    for _ in range(2):
        a, b = scaled(*few.backward_np()), scaled(*full.backward_np())
        assert np.abs(a - b).max() <= 1e-5 * np.abs(b).max()


def test_default_keeps_steps_when_memory_is_ample(pkg):  # noqa: F811
    eng = engine(pkg, 100, 30, None)
    assert eng.ws.numel() == engine(pkg, 100, 30, True).ws.numel()
