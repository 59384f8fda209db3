"""Held particles set to new poses after fixed-geometry steps, which bin nothing:
the next step refills the nodes they leave.  The particles jump several nodes in
y and z, out of their old bricks (4x2 nodes there), so those are not listed
again; the near set is a large share of the box, so that the plain sweep runs
beside the flag pass.  Expected, to the bit: the same particles not declared
fixed (no DEM sub-steps), which run the brick sweeps throughout; and each new
fluid node counted once."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts
    pytest.skip("no CUDA device", allow_module_level=True)

# poses of two spheres of radius 5 and 4 (one stays), the last ones far from the first
POSES = [[(14.3, 11.2, 10.1), (30.2, 25.3, 34.4)], [(14.3, 20.7, 17.6), (30.2, 25.3, 34.4)],
         [(15.1, 33.4, 33.2), (30.2, 12.1, 12.3)]]


@pytest.fixture(scope="module")
def pkg():
    from paper_2206_11634_gb300 import build as b
    b.build()
    import paper_2206_11634_gb300 as p
    return p


def spheres(pkg, pose, fixed=1):
    return [pkg.make_particle([[0, 0, 0]], [r * r], x, v=(0.01, 0.0, -0.004), fixed=fixed, mass=100.0,
                              inertia=np.eye(3) * 1e3) for x, r in zip(POSES[pose], (5.0, 4.0))]


KW = dict(periodic=(1, 1, 1), tau=0.7, force=(1e-5, 0.0, -2e-6), max_particles=2)


def flow(Q, n, seed=3):
    from tests.test_gpu_static import pkg_weight
    g = torch.Generator(device="cuda").manual_seed(seed)
    w = torch.tensor([pkg_weight(Q, i) for i in range(Q)], dtype=torch.float64, device="cuda")
    return w[:, None, None, None] * (1.0 + 0.02 * (torch.rand((Q, n, n, n), generator=g, device="cuda",
                                                              dtype=torch.float64) - 0.5))


def states(lat):
    c = lat.counters()
    return (lat.populations().cpu().numpy(), lat.flags().cpu().numpy(), *lat.forces(), c["nlinks"], c["nrefill"],
            c["near_bricks"])


@pytest.mark.parametrize("storage,Q", [("f32", 19), ("f16", 15)])
@pytest.mark.parametrize("n", [40, 45])
@pytest.mark.parametrize("held", [4, 5, 10, 11, 12])  # 3 brick steps, then 1, 2, 7, 8, 9 fixed-geometry ones
def test_lattice(pkg, storage, Q, n, held):
    runs = []
    for fixed in (1, 0):
        lat = pkg.Lattice(n, n, n, storage=storage, lattice=Q, **KW)
        lat.set_populations(flow(Q, n))
        out = []
        for pose in range(len(POSES)):
            lat.set_particles(spheres(pkg, pose, fixed))
            lat.step(1)
            out.append(states(lat))
            lat.step(held - 1)
            out.append(states(lat)[:-1])  # (fixed-geometry steps have no near bricks to count)
        runs.append(out)
    assert runs[0][2][5] > 300  # the sphere of radius 5 left its nodes
    for a, b in zip(*runs):
        for x, y in zip(a, b):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("held", [4, 5, 10, 11, 12])
def test_batch(pkg, storage, held):
    sides = (40, 45)
    bt = pkg.Batch([dict(nx=n, ny=n, nz=n, storage=storage, n_sub=0, **KW) for n in sides])
    single = []
    for n in sides:
        single.append(pkg.Lattice(n, n, n, storage=storage, **KW))
    for pose in range(len(POSES)):
        for c in range(2):
            at = pose if c == 0 else 0  # the second box's spheres stay
            bt.set_particles(c, spheres(pkg, at))
            single[c].set_particles(spheres(pkg, at, 0))
        for steps in (1, held - 1):
            bt.step(steps)
            for c, lat in enumerate(single):
                lat.step(steps)
                assert np.array_equal(bt.populations(c).cpu().numpy(), lat.populations().cpu().numpy())
                for x, y in zip(bt.forces(c), lat.forces()):
                    assert np.array_equal(x, y)


def test_held_particles_with_dem_sub_steps(pkg):
    """The DEM runs behind the fixed-geometry kernels of each step: two held
    spheres that overlap have the contact load of the first step (brick sweeps) in
    every later one (FP32 contact geometry, its overlap to 1e-6 of 0.5), and the
    flow keeps the bits of a run without DEM."""
    pops = []
    for n_sub in (0, 10):
        lat = pkg.Lattice(40, 40, 40, n_sub=n_sub, kn=100.0, kt=50.0, **KW)
        lat.set_populations(flow(19, 40))
        lat.set_particles([pkg.make_particle([[0, 0, 0]], [16.0], (14.0 + 9.5 * k, 20.0, 20.0), Rs=1.0, fixed=1,
                                             mass=100.0, inertia=np.eye(3) * 1e3) for k in range(2)])
        load = []
        for steps in (1, 1, 7, 1, 5):
            lat.step(steps)
            load.append(lat.contact_forces()[0])
        pops.append(lat.populations().cpu().numpy())
        assert (np.abs(load[0][:, 0]).min() > 1.0) == (n_sub > 0)
        for F in load:
            assert np.abs(F - load[0]).max() <= 1e-5 * np.abs(load[0]).max()
    assert np.array_equal(*pops)
