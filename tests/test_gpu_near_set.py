"""The bricks the flag pass and the near sweep look at: of those a particle's
search box meets, the ones M can reach c0 in.  Flags against M evaluated at
every node in FP64, links counted from the flags; FP64 forces of a particle
that leaves its bricks against those of the FP32 sweep, which keeps no
per-brick sums."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts
    pytest.skip("no CUDA device", allow_module_level=True)

E19 = [(x, y, z) for x in (-1, 0, 1) for y in (-1, 0, 1) for z in (-1, 0, 1) if 0 < abs(x) + abs(y) + abs(z) < 3]


@pytest.fixture(scope="module")
def pkg():
    from paper_2206_11634_gb300 import build as b
    b.build()
    import paper_2206_11634_gb300 as p
    return p


def rotation(rng):
    q = rng.normal(size=4)
    q /= np.linalg.norm(q)
    w, x, y, z = q
    return q, np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
                        [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
                        [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]])


def owners(shape, periodic, parts, c0):
    nz, ny, nx = shape
    grid = np.stack(np.meshgrid(np.arange(nx), np.arange(ny), np.arange(nz), indexing="ij"), -1).astype(float)
    best, own, gap = np.zeros((nx, ny, nx * 0 + nz)), np.full((nx, ny, nz), 0), np.inf
    for j, (cp, K) in enumerate(parts):
        M = np.zeros((nx, ny, nz))
        for c, k in zip(cp, K):
            d = grid - c
            for a, L in enumerate((nx, ny, nz)):
                if periodic[a]:
                    d[..., a] -= L * np.floor(d[..., a] / L + 0.5)
            M += k / (d ** 2).sum(-1)
        gap = min(gap, np.abs(M - c0).min())
        new = (M >= c0) & (M > best)
        own[new] = j + 1
        best[new] = M[new]
    return own.transpose(2, 1, 0), gap


@pytest.mark.parametrize("storage", ["f64", "f32", "f16"])
@pytest.mark.parametrize("c0", [1.0, 0.3])
@pytest.mark.parametrize("periodic", [(1, 1, 1), (0, 1, 0), (0, 0, 0)])
def test_flags_and_links(pkg, storage, c0, periodic):
    nx, ny, nz = 75, 50, 41  # ragged bricks along every axis
    rng = np.random.default_rng(5)
    for trial in range(6):
        parts, ps = [], []
        for j in range(7):
            n = int(rng.integers(1, 17))
            cp = rng.normal(size=(n, 3)) * rng.uniform(0.3, 3.0)  # compact and far-flung control points
            cp[:, 0] *= rng.uniform(0.2, 3.0)
            cp -= cp.mean(0)
            K = rng.uniform(0.0, 2.0, n) * rng.uniform(0.1, 3.0) / n * 4 * c0
            x = rng.uniform(0, 1, 3) * (nx - 1, ny - 1, nz - 1)
            q, R = rotation(rng)
            parts.append((cp @ R.T + x, K))
            ps.append(pkg.make_particle(cp, K, tuple(x), q=tuple(q), fixed=1, mass=1.0, inertia=np.eye(3)))
        want, gap = owners((nz, ny, nx), periodic, parts, c0)
        assert gap > 1e-11
        if trial == 0:  # the later trials replace the particles (bricks left behind)
            lat = pkg.Lattice(nx, ny, nz, storage=storage, periodic=periodic, tau=0.8, max_particles=7, c0=c0)
        lat.set_particles(ps)
        lat.step(1)
        assert np.array_equal(lat.flags().cpu().numpy(), want)
        fluid, solid, links = want == 0, want > 0, 0
        for e in E19:
            s = np.roll(solid, (-e[2], -e[1], -e[0]), (0, 1, 2))
            for a, c in ((0, e[2]), (1, e[1]), (2, e[0])):
                if c and not periodic[2 - a]:
                    sl = [slice(None)] * 3
                    sl[a] = -1 if c > 0 else 0
                    s[tuple(sl)] = False
            links += int((fluid & s).sum())
        assert lat.counters()["nlinks"] == links


def test_fp64_forces_of_a_moving_particle(pkg):
    """A sphere moves by half a node a step for 30 steps, so that bricks with
    links become link-free ones of its search box.  Both lattices start from
    the same populations; FP32's differences from FP64's (2^-24 of populations
    of order w_i per link and step, some 600 links, 30 steps) stay under 1e-4
    of the largest force, a brick's share of it is some 1e-2."""
    F = {}
    for storage in ("f64", "f32"):
        lat = pkg.Lattice(64, 36, 36, storage=storage, periodic=(1, 1, 1), tau=0.8, max_particles=1)
        F[storage] = []
        for k in range(30):
            lat.set_particles([pkg.make_particle([[0, 0, 0]], [30.0], (20.3 + 0.5 * k, 13.1 + 0.3 * k, 12.2 + 0.4 * k),
                                                 fixed=1, v=(0.05, 0.03, 0.04), mass=1.0, inertia=np.eye(3))])
            lat.step(1)
            f, t = lat.forces()
            F[storage].append(np.concatenate([np.ravel(f), np.ravel(t)]))
    a, b = np.array(F["f64"]), np.array(F["f32"])
    assert np.abs(a - b).max() < 1e-4 * np.abs(a).max()
