"""The fixed-geometry sweep's two kernels as programmatic dependent launches:
the same bits as the brick sweeps (the same particles not declared fixed, no
DEM sub-steps), for few and for many link nodes (four and eight of them a warp),
warps that meet several particles, walls and ragged boxes; and the same bits
whether the steps run back to back or one at a time with the device idle in
between.  The arithmetic is shared, so equality is exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts
    pytest.skip("no CUDA device", allow_module_level=True)

BOXES = {
    # one small sphere; its link nodes are few (four a warp)
    "small": (21, 17, 19, (1, 1, 1), [(10.3, 8.2, 9.1, 4.0)]),
    # 18 000 link nodes: more than every resident warp holds four of
    "large": (79, 75, 77, (1, 1, 1), [(39.2, 37.4, 38.1, 31.0)]),
    # five small spheres, two of them overlapping, against walls
    "five": (47, 37, 33, (1, 0, 0), [(8.1, 8.3, 5.2, 5.0), (20.2, 9.4, 6.1, 5.0), (27.6, 11.0, 7.3, 5.5),
                                     (40.1, 30.2, 27.9, 4.5), (3.0, 28.5, 20.2, 4.0)]),
}


@pytest.fixture(scope="module")
def pkg():
    from paper_2206_11634_gb300 import build as b
    b.build()
    import paper_2206_11634_gb300 as p
    return p


def lattice(pkg, box, storage, Q, fixed, seed=3):
    nx, ny, nz, per, balls = BOXES[box]
    lat = pkg.Lattice(nx, ny, nz, storage=storage, lattice=Q, periodic=per, tau=0.7, force=(1e-5, 0.0, -2e-6),
                      max_particles=len(balls))
    lat.set_particles([pkg.make_particle([[0, 0, 0], [0.6, 0, 0]], [0.5 * r * r, 0.5 * r * r], (x, y, z), fixed=fixed,
                                         v=(0.01, 0, 0.004), w=(0, 1e-3, 0), mass=100.0, inertia=np.eye(3) * 1e3)
                       for x, y, z, r in balls])
    g = torch.Generator(device="cuda").manual_seed(seed)
    w = torch.tensor([pkg_weight(Q, i) for i in range(Q)], dtype=torch.float64, device="cuda")
    lat.set_populations(w[:, None, None, None]
                        * (1.0 + 0.02 * (torch.rand((Q, nz, ny, nx), generator=g, device="cuda",
                                                    dtype=torch.float64) - 0.5)))
    return lat


def pkg_weight(Q, i):
    if Q == 19:
        return 1 / 3 if i == 0 else (1 / 18 if i <= 6 else 1 / 36)
    return 2 / 9 if i == 0 else (1 / 9 if i <= 6 else 1 / 72)


def state(lat):
    return (lat.populations().cpu().numpy(), *lat.forces(), lat.counters()["nlinks"])


@pytest.mark.parametrize("box", list(BOXES))
@pytest.mark.parametrize("storage,Q", [("f32", 19), ("f32", 15), ("f16", 19)])
def test_same_bits_as_the_brick_sweeps(pkg, box, storage, Q):
    runs = []
    for fixed in (1, 0):
        lat = lattice(pkg, box, storage, Q, fixed)
        lat.step(9)
        runs.append(state(lat))
    (f1, F1, T1, n1), (f0, F0, T0, n0) = runs
    assert n1 == n0 and n1 > 0
    assert np.array_equal(f1, f0)
    assert np.array_equal(F1, F0) and np.array_equal(T1, T0)


@pytest.mark.parametrize("box", list(BOXES))
def test_back_to_back_steps_same_bits(pkg, box):
    a, b = lattice(pkg, box, "f32", 19, 1), lattice(pkg, box, "f32", 19, 1)
    a.step(40)
    for _ in range(40):
        b.step(1)
        torch.cuda.synchronize()
    for x, y in zip(state(a), state(b)):
        assert np.array_equal(x, y)


def test_batch_particles_set_again(pkg):
    """A batch whose particles are set again after an odd number of
    fixed-geometry steps (which do not advance the brick sweeps' step counters):
    the same bits as single lattices through the same calls."""
    def held(n, shift):
        return pkg.make_particle([[0, 0, 0], [1.0, 0.5, 0]], [8.0, 9.0], (n / 2 + shift, n / 2 - 0.3, n / 2 + 0.1),
                                 fixed=1, mass=1.0, inertia=np.eye(3))
    sizes = [24, 33, 29]
    kw = [dict(nx=n, ny=n, nz=n, storage="f32", periodic=(1, 1, 1), tau=0.8, force=(1e-5, 0, 0), n_sub=0,
               max_particles=1) for n in sizes]
    bt = pkg.Batch(kw)
    singles = [pkg.Lattice(k["nx"], k["ny"], k["nz"], **{a: v for a, v in k.items() if a not in ("nx", "ny", "nz")})
               for k in kw]
    for shift, calls in ((0.2, (3, 4, 1)), (0.9, (1, 6, 17, 2)), (-0.4, (20,))):
        for c, n in enumerate(sizes):
            bt.set_particles(c, [held(n, shift)])
            singles[c].set_particles([held(n, shift)])
        for k in calls:
            bt.step(k)
            for lat in singles:
                lat.step(k)
        for c, lat in enumerate(singles):
            assert np.array_equal(bt.populations(c).cpu().numpy(), lat.populations().cpu().numpy())
            for a, b in zip(bt.forces(c), lat.forces()):
                assert np.array_equal(a, b)


@pytest.mark.parametrize("storage,Q", [("f32", 19), ("f32", 15), ("f16", 19), ("bf16", 15)])
def test_many_near_bricks_same_bits(pkg, monkeypatch, storage, Q):
    # about 9 700 near bricks expected: beyond the count from which the near
    # sweep runs four CTAs per SM instead of two
    monkeypatch.setitem(BOXES, "many", (97, 89, 91, (1, 0, 1), [
        (16.2 + 32.1 * i, 14.7 + 29.3 * j, 23.1 + 45.2 * k, 13.0 + 0.2 * i)
        for i in range(3) for j in range(3) for k in range(2)]))
    runs = []
    for fixed in (1, 0):
        lat = lattice(pkg, "many", storage, Q, fixed)
        lat.step(5)
        runs.append(state(lat))
    (f1, F1, T1, n1), (f0, F0, T0, n0) = runs
    assert n1 == n0 and n1 > 0
    assert np.array_equal(f1, f0)
    assert np.array_equal(F1, F0) and np.array_equal(T1, T0)
