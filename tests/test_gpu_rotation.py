"""A free particle's rotation over one step on the GPU: FP32 pairs where they
carry FP64's accuracy (dem_rot32.cuh), FP64 sub-steps elsewhere, chosen per
particle.  Expected: the sub-steps by numpy in FP64 from the torque that the
GPU reports for the step.

Tolerance 1e-13: 333 FP64 sub-steps of about six roundings each, 2^-53 of the
state at most, add up to 2e-13 in the worst direction and ten times less in
practice; the reported w is rotated once more."""
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


@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("n_sub", [1, 7, 8, 100, 333])
def test_free_rotation_per_particle(pkg, storage, n_sub):
    from perf.cases import _turn
    rng = np.random.default_rng(5)
    # 11 particles: two warps of quads, one ragged; slow, fast (past the pairs'
    # limit), at rest and held ones side by side
    speed = [1e-5, 2e-3, 8e-2, 0.0, 5e-3, 6.2e-3, 1e-3, 0.3, 3e-4, 0.0, 2e-3]
    parts = []
    for k, s in enumerate(speed):
        w = rng.normal(size=3)
        m = rng.uniform(1.0, 2.0, 3)
        A = np.linalg.qr(rng.normal(size=(3, 3)))[0]
        inertia = A @ np.diag([m[0] + m[1], m[1] + m[2], m[2] + m[0]]) @ A.T * 4e3
        q = rng.normal(size=4)
        parts.append(dict(cp=rng.uniform(-1, 1, (2, 3)), K=np.array([5.0, 6.0]),
                          x=np.array([8.0 + 14 * (k % 4), 8.0 + 14 * (k // 4), 11.3]), q=q / np.linalg.norm(q),
                          v=np.zeros(3), w=s * w / np.linalg.norm(w), mass=200.0,
                          inertia=0.5 * (inertia + inertia.T), fixed=int(k == 6)))
    lat = pkg.Lattice(58, 44, 24, storage=storage, periodic=(1, 1, 1), n_sub=n_sub, tau=0.8, u0=(0.02, -0.01, 0.015),
                      max_particles=len(parts), kn=100.0, kt=50.0)
    lat.set_particles([pkg.make_particle(p["cp"], p["K"], p["x"], q=p["q"], v=p["v"], w=p["w"], density=1.5,
                                         mass=p["mass"], inertia=p["inertia"], fixed=p["fixed"]) for p in parts])
    lat.step(1)
    _, T = lat.forces()
    got = lat.particles()
    assert np.abs(T).max() > 1e-3
    for p, t, s in zip(parts, T, got):
        q, w = (p["q"], p["w"]) if p["fixed"] else _turn(p, t, n_sub)
        scale = max(np.linalg.norm(w), 1e-9)
        assert np.abs(s["q"] * np.sign(s["q"] @ q) - q).max() <= 1e-13
        assert np.abs(s["w"] - w).max() <= 1e-13 * scale
