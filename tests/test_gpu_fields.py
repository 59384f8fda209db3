"""Macroscopic fields and stored populations read out in FP64 (lbm_get_fields,
lbm_get_populations): lattices below FP64 sum a node's FP32 offsets exactly
and convert without FP64 arithmetic.

The expected values are exact sums (Python fractions of the stored FP32
offsets).  Tolerances: the density is one rounding of the momentum-free sum
and one of the addition of rho0 (2^-53 of rho0 each); a velocity component is
one rounding of the exact momentum, the quotient by the rounded density
(2^-53 each) and the rounding of the quotient within 0.51 ulp: 4 x 2^-53
relative.  A node whose offsets span more than 2^30 may lose bits below 2^-53
of the largest offset on each of them: 19 x 2^-53 of it, absolute."""
from fractions import Fraction

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


def directions(Q):
    from perf.cases import _lattice_vectors
    return _lattice_vectors(Q)


def offsets(rng, storage, Q, shape, w, spread):
    """Populations and the FP32 offsets g = f - w that they are stored as.
    FP32: offsets of every size down to 10^-spread.  16 bits: g = w s with s on
    the type's own grid in 2^-6..2^-3, which f / w - 1 in FP32 rounds back to."""
    w32 = np.array(w, dtype=np.float32)[:, None, None, None]
    if storage == "f32":
        f = w32.astype(np.float64) * (1.0 + rng.normal(size=(Q,) + shape) * 10.0 ** rng.uniform(-spread, -1.5,
                                                                                               (Q,) + shape))
        return f, f.astype(np.float32) - w32
    s = rng.choice([-1.0, 1.0], (Q,) + shape) * 2.0 ** rng.uniform(-6, -3, (Q,) + shape)
    s = torch.from_numpy(s).to(torch.float16 if storage == "f16" else torch.bfloat16).float().numpy()
    return w32.astype(np.float64) * (1.0 + s.astype(np.float64)), w32 * s


@pytest.mark.parametrize("Q", [19, 15])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("force", [(0.0, 0.0, 0.0), (3e-6, 0.0, -2e-5)])
def test_fields_are_the_exact_sums(pkg, Q, storage, force):
    e, w = directions(Q)
    w = np.array(w)
    rng = np.random.default_rng(11)
    nx, ny, nz = 33, 5, 3  # one node past a warp
    lat = pkg.Lattice(nx, ny, nz, lattice=Q, storage=storage, periodic=(1, 1, 1), force=force)
    f, g = offsets(rng, storage, Q, (nz, ny, nx), w, 7.0)
    # rest: every offset zero, or in 16 bits the rounding of w (1/w) - 1
    w32 = np.array(w, dtype=np.float32)
    f[:, 0, 0, :4] = w32[:, None]
    rest = (w32.astype(np.float64) * (np.float32(1.0) / w32).astype(np.float64) - 1.0).astype(np.float32)
    if storage != "f32":
        rest = torch.from_numpy(rest).to(torch.float16 if storage == "f16" else torch.bfloat16).float().numpy()
        g[:, 0, 0, :4] = (w32 * rest)[:, None]
    else:
        g[:, 0, 0, :4] = 0.0
    lat.set_populations(torch.from_numpy(f))
    rho, u, _ = lat.fields()
    rho, u = rho.cpu().numpy(), u.cpu().numpy()
    eps = 2.0 ** -53
    bad = 0
    for z in range(nz):
        for y in range(ny):
            for x in range(nx):
                v = [Fraction(float(g[i, z, y, x])) for i in range(Q)]
                top = max(abs(float(t)) for t in v)
                r = Fraction(1) + sum(v)
                slack = 19 * eps * top
                assert abs(rho[z, y, x] - float(r)) <= 2.0 * eps * float(r) + slack
                for a in range(3):
                    m = sum(e[i][a] * v[i] for i in range(Q)) - Fraction(force[a]) / 2
                    ua = float(m / r)
                    # the half force is subtracted in FP64: one rounding more, of the momentum
                    tol = 4.0 * eps * (abs(ua) + 0.5 * abs(force[a])) + slack
                    bad += abs(u[a, z, y, x] - ua) > tol
    assert bad == 0


def test_fields_not_finite(pkg):
    """A population that is not finite leaves its node's fields not finite."""
    e, w = directions(19)
    f = np.tile(np.array(w)[:, None, None, None], (1, 2, 2, 34))
    f[3, 0, 0, 5] = np.inf
    f[7, 1, 1, 33] = np.nan
    lat = pkg.Lattice(34, 2, 2, storage="f32", periodic=(1, 1, 1))
    lat.set_populations(torch.from_numpy(f))
    rho, u, _ = lat.fields()
    hit = np.zeros((2, 2, 34), bool)
    hit[0, 0, 5] = hit[1, 1, 33] = True
    assert np.array_equal(~np.isfinite(rho.cpu().numpy()), hit)
    assert np.array_equal(~np.isfinite(u[0].cpu().numpy()), hit)


def test_population_round_trip(pkg):
    """set_populations rounds to FP32 like the cast and get_populations widens
    like it, over FP32's whole range (subnormals, overflow to infinity)."""
    e, w = directions(19)
    rng = np.random.default_rng(12)
    shape = (2, 3, 65)
    f = rng.normal(size=(19,) + shape) * 10.0 ** rng.uniform(-44, 37, (19,) + shape)
    ties = (np.arange(65) + 0.5) * 2.0 ** -23 + 1.0   # halfway between FP32 neighbours
    f[0, 0, 0] = ties
    f[1, 0, 0] = np.nextafter(ties, 2.0)
    f[2, 0, 0, :4] = [3.5e38, -3.5e38, 0.0, 1e-46]
    lat = pkg.Lattice(65, 3, 2, storage="f32", periodic=(1, 1, 1))
    lat.set_populations(torch.from_numpy(f))
    w32 = np.array(w, dtype=np.float32)[:, None, None, None]
    with np.errstate(over="ignore"):
        want = w32 + (f.astype(np.float32) - w32)  # w rho0 is exact with rho0 = 1
    assert np.array_equal(lat.populations().cpu().numpy(), want.astype(np.float64))


@pytest.mark.parametrize("storage", ["f16", "bf16"])
def test_population_round_trip_16_bit(pkg, storage):
    e, w = directions(19)
    f, g = offsets(np.random.default_rng(13), storage, 19, (2, 3, 65), w, 0.0)
    lat = pkg.Lattice(65, 3, 2, storage=storage, periodic=(1, 1, 1))
    lat.set_populations(torch.from_numpy(f))
    w32 = np.array(w, dtype=np.float32)[:, None, None, None]
    s = np.round(g / w32 * 2.0 ** 18) / 2.0 ** 18  # the grid value (at most 11 bits below 2^-3)
    want = (w32 * (np.float32(1.0) + s.astype(np.float32))).astype(np.float64)
    assert np.array_equal(lat.populations().cpu().numpy(), want)
