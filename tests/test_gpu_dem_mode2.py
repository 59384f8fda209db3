"""dem_mode 2 (LBM_DEM_FP64_ALL) runs the rotation sub-steps of free particles in
FP64, as its name says; the default mode may run them in FP32 pairs
(dem_rot32.cuh).  Both modes run the same kernel on an FP64 lattice, from the same
load, so bits that agree mean the same arithmetic: with fewer than 8 sub-steps
both are FP64, and with 100 for a body whose half angle a sub-step, |w| / 200, is
over 2^-16 (rot32_applies).  The slower ones' last bits differ, and only those:
1e-13 of the state, the tolerance of tests/test_gpu_rotation.py."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.fixture(scope="module")
def pkg():
    from paper_2206_11634_gb300 import build as b
    b.build()
    import paper_2206_11634_gb300 as p
    return p


def turned(pkg, mode, n_sub, storage):
    rng = np.random.default_rng(8)
    lat = pkg.Lattice(58, 44, 24, storage=storage, periodic=(1, 1, 1), n_sub=n_sub, tau=0.8, max_particles=12,
                      kn=100.0, kt=50.0, dem_mode=mode)
    parts, speed = [], []
    for k in range(12):
        m = rng.uniform(1.0, 2.0, 3)
        inertia = np.diag([m[0] + m[1], m[1] + m[2], m[2] + m[0]]) * 4e3
        q = rng.normal(size=4)
        w = 3e-3 * rng.normal(size=3)
        speed.append(np.linalg.norm(w))
        parts.append(pkg.make_particle([[0.4, 0.0, 0.1], [-0.4, 0.0, -0.1]], [5.0, 6.0],
                                       (8.0 + 14 * (k % 4), 8.0 + 14 * (k // 4), 11.3), q=q / np.linalg.norm(q),
                                       w=w, density=1.5, mass=200.0, inertia=inertia))
    lat.set_particles(parts)
    lat.step(1)
    slow = np.array(speed) <= 200 * 2.0 ** -16
    assert 0 < slow.sum() < 12
    return np.array([np.concatenate([s["q"], s["w"]]) for s in lat.particles()]), slow


@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("n_sub", [7, 100])
def test_rotation_of_mode_2(pkg, n_sub, storage):
    (a, slow), (b, _) = turned(pkg, 2, n_sub, storage), turned(pkg, 0, n_sub, storage)
    assert np.array_equal((a != b).any(axis=1), slow if n_sub >= 8 else np.zeros(12, bool))
    assert np.abs(a[:, :4] - b[:, :4]).max() <= 1e-13
    assert np.abs(a[:, 4:] - b[:, 4:]).max() <= 1e-13 * np.linalg.norm(b[:, 4:], axis=1).max()
