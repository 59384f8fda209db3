"""A batch whose recorded geometry does not fit (one box crowded with spheres)
keeps the brick sweeps: sixteen steps at a time as replays of a captured graph, the
rest launched directly, with the step numbers in device counters.  Expected, to
the bit: each box stepped alone with particles not declared fixed, whatever the
split of the steps into calls, and after new poses."""
import itertools

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts
    pytest.skip("no CUDA device", allow_module_level=True)

from tests.test_gpu_set_again import pkg  # noqa: E402,F401

KW = dict(periodic=(1, 1, 1), tau=0.7, force=(1e-5, 0.0, -2e-6), n_sub=0)


def crowd(pkg, n, per_axis, radius, shift, fixed):  # noqa: F811
    at = (np.arange(per_axis) + 0.5) * n / per_axis
    return [pkg.make_particle([[0, 0, 0]], [radius * radius], np.array(c) + shift, v=(0.004, 0.0, -0.002), fixed=fixed,
                              mass=50.0, inertia=np.eye(3) * 400.0) for c in itertools.product(at, at, at)]


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("calls", [(1, 20, 16, 33), (40, 1, 16), (3, 16, 48), (70,)])
def test_brick_steps_of_a_crowded_batch(pkg, storage, calls):  # noqa: F811
    boxes = [(40, 3, 5.2), (45, 1, 6.0)]  # 27 spheres (more than 16 384 links), one sphere
    batch = pkg.Batch([dict(nx=n, ny=n, nz=n, storage=storage, max_particles=k ** 3, **KW) for n, k, _ in boxes])
    single = [pkg.Lattice(n, n, n, storage=storage, max_particles=k ** 3, **KW) for n, k, _ in boxes]
    alone = pkg.Lattice(40, 40, 40, storage=storage, max_particles=27, **KW)
    alone.set_particles(crowd(pkg, *boxes[0], 0.0, 1))
    alone.step(5)
    assert b"brick sweeps kept" in alone.L.lbm_last_error(alone.h)
    for shift in (0.0, (0.7, 3.1, 2.4)):
        for c, box in enumerate(boxes):
            batch.set_particles(c, crowd(pkg, *box, shift, 1))
            single[c].set_particles(crowd(pkg, *box, shift, 0))
        for steps in calls:
            batch.step(steps)
            for c, lat in enumerate(single):
                lat.step(steps)
                assert np.array_equal(batch.populations(c).cpu().numpy(), lat.populations().cpu().numpy())
                for x, y in zip(batch.forces(c), lat.forces()):
                    assert np.array_equal(x, y)


def test_captured_fixed_steps_replay(pkg):  # noqa: F811
    """An even number of fixed-geometry steps in a caller's own graph: five
    replays are ten steps."""
    stream = torch.cuda.Stream()
    runs = []
    for captured in (True, False):
        b = pkg.Batch([dict(nx=n, ny=n, nz=n, storage="f32", max_particles=1, **KW) for n in (32, 45)], stream=stream)
        for c, n in enumerate((32, 45)):
            b.set_particles(c, crowd(pkg, n, 1, 5.0, 0.3, 1))
        b.step(6)
        torch.cuda.synchronize()
        if captured:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                b.step(2)
            for _ in range(5):
                graph.replay()
        else:
            b.step(10)
        torch.cuda.synchronize()
        runs.append([x for c in range(2) for x in (b.populations(c).cpu().numpy(), *b.forces(c))])
    for x, y in zip(*runs):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("held", [3, 4, 5, 6])  # 4: the step that tries to record the geometry is the last
def test_crowded_lattice_set_again(pkg, held):  # noqa: F811
    """A single lattice whose geometry does not fit: new poses right after the
    step that found so, and around it, against particles not declared fixed."""
    runs = []
    for fixed in (1, 0):
        lat = pkg.Lattice(40, 40, 40, storage="f32", max_particles=27, **KW)
        out = []
        for shift in (0.0, (0.7, 4.1, 5.4), (0.2, 1.3, 2.0)):
            lat.set_particles(crowd(pkg, 40, 3, 5.2, shift, fixed))
            for steps in (1, held - 1):
                lat.step(steps)
                out += [lat.populations().cpu().numpy(), lat.flags().cpu().numpy(), *lat.forces(),
                        lat.counters()["nrefill"]]
        runs.append(out)
    for x, y in zip(*runs):
        assert np.array_equal(x, y)
