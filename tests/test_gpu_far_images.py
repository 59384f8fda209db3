"""Particles whose positions lie many box lengths away along periodic axes (the
library does not wrap them): an FP64 lattice classifies its nodes as for the
image inside the box.  Their FP32 positions are too coarse there, so neither the
flag pass's FP32 decision nor the binning's FP32 bound may rest on them.

Expected flags: M at every node in FP64 for the image in the box.  A position
shifted by s is rounded to 2^-53 s, under 2^-32 for the largest shift here, which
moves M near the surface (|grad M| of order c0) by less than 1e-8; no node lies
within 1e-6 of it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts
    pytest.skip("no CUDA device", allow_module_level=True)

from tests.test_gpu_near_set import owners, pkg, rotation  # noqa: E402,F401


@pytest.mark.parametrize("lengths", [0, 3, 40, -2 ** 9, 2 ** 14, -2 ** 15])
@pytest.mark.parametrize("periodic", [(1, 1, 1), (1, 0, 1)])
def test_flags_of_far_images(pkg, lengths, periodic):  # noqa: F811
    nx, ny, nz = 70, 36, 33
    rng = np.random.default_rng(17)
    for trial in range(8):
        parts, ps = [], []
        for j in range(5):
            n = int(rng.integers(1, 6))
            cp = rng.normal(size=(n, 3)) * 1.5
            cp -= cp.mean(0)
            K = rng.uniform(1.0, 20.0, n) / n
            x = rng.uniform(0, 1, 3) * (nx - 1, ny - 1, nz - 1)
            q, R = rotation(rng)
            parts.append((cp @ R.T + x, K))
            far = x + lengths * np.array(periodic) * (nx, ny, nz)
            ps.append(pkg.make_particle(cp, K, tuple(far), q=tuple(q), fixed=1, mass=1.0, inertia=np.eye(3)))
        want, gap = owners((nz, ny, nx), periodic, parts, 1.0)
        assert gap > 1e-6
        if trial == 0:
            lat = pkg.Lattice(nx, ny, nz, storage="f64", periodic=periodic, tau=0.8, max_particles=5)
        lat.set_particles(ps)
        lat.step(1)
        assert np.array_equal(lat.flags().cpu().numpy(), want)
