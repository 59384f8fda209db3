"""The drag gradient where the adjoint's variants can go wrong: runs that keep
every step's data and runs that keep checkpoints, box sides that are no
multiple of a span or a warp, a particle without links, no body force.

A 176^3 run of 100 steps would keep 8.7 GB of steps, above the limit for
keeping all, and keeps checkpoints: its gradient is compared along itself with
a central difference of its own forward run, as the full-size test of
tests/test_gpu_adjoint.py does (h = 2e-3, 1e-2: some links cross q = 1/2)."""
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


def engine(pkg, shape, cp, K, T, W, force=(4e-6, 1e-6, 0.0), u0=(0.0, 0.0, 0.0)):
    from paper_2206_11634_gb300.adjoint import AdjointDrag
    c = np.mean(cp, axis=0)
    p = pkg.make_particle(np.asarray(cp) - c, K, c, fixed=1, mass=1.0, inertia=np.eye(3))
    return AdjointDrag(*shape, particle=p, T=T, W=W, tau=0.8, u0=u0, force=force)


CP = np.array([[15.2, 15.8, 15.1], [17.9, 14.6, 16.3], [14.1, 17.2, 17.0]])
K = np.array([6.0, 5.0, 4.0])


def scaled(g_cp, g_K):
    return np.concatenate([np.ravel(g_cp), g_K * K])


def test_run_with_checkpoints(pkg):
    from paper_2206_11634_gb300 import workloads as W
    case = W.adjoint_case(n=176, ncp=4, T=100, W=20)
    cp, Kc = case["cp_world"], case["K"]
    eng = engine(pkg, (176, 176, 176), cp, Kc, 100, 20, case["force"], case["u0"])
    assert eng.ws.numel() < 8 << 30  # it keeps checkpoints
    eng.forward_np(cp, Kc)
    g_cp, g_K = eng.backward_np()
    v = np.concatenate([np.ravel(g_cp), g_K * Kc])
    d = v / np.linalg.norm(v)
    h = 2e-3
    n = 3 * len(Kc)
    Jp = eng.forward_np(cp + h * d[:n].reshape(-1, 3), Kc * (1 + h * d[n:]))
    Jm = eng.forward_np(cp - h * d[:n].reshape(-1, 3), Kc * (1 - h * d[n:]))
    fd = (Jp - Jm) / (2 * h)
    assert abs(fd - np.linalg.norm(v)) <= 1e-2 * abs(fd)


@pytest.mark.parametrize("shape", [(32, 32, 32), (33, 35, 31), (64, 29, 34), (37, 32, 43)])
@pytest.mark.parametrize("force", [(4e-6, 1e-6, 0.0), (0.0, 0.0, 0.0)])
def test_gradient_against_autograd_in_fp64(pkg, shape, force):
    """Every component within 1e-4 of the largest one of the FP64 gradient by
    plain torch autograd (the tolerance of tests/test_gpu_adjoint.py), J within
    1e-4 relative."""
    from perf import cases as M
    T, W = 24, 9
    u0 = (0.02, 0.005, -0.003)
    eng = engine(pkg, shape, CP, K, T, W, force, u0)
    J = eng.forward_np(CP, K)
    g = scaled(*eng.backward_np())
    Jx, gx = fp64_gradient(M, shape, T, W, force, u0)
    assert abs(J - Jx) <= 1e-4 * abs(Jx)
    assert np.abs(g - gx).max() <= 1e-4 * np.abs(gx).max()


def fp64_gradient(M, shape, T, W, force, u0):
    nx, ny, nz = shape
    R = M.Reference((nz, ny, nx), 19, (1, 1, 1), 0.8, force)
    c = CP.mean(axis=0)
    with torch.no_grad():
        R.set_particles([dict(cp=CP - c, K=K, x=c, v=np.zeros(3), w=np.zeros(3), q=np.array([1.0, 0, 0, 0]))])
        own = R.classify()
        R.own = own
        i, nn, j, _, ff, ok, arm = R.find_links(own)
    cp = torch.tensor(CP, device="cuda").requires_grad_(True)
    Kt = torch.tensor(K, device="cuda").requires_grad_(True)
    R.cp, R.K = cp[None], Kt[None]
    q = R.fraction(j, R.position(nn).double(), -R.E[i])
    u = torch.tensor(u0, dtype=torch.float64, device="cuda").expand(nz, ny, nx, 3)
    one = torch.ones((nz, ny, nx), dtype=torch.float64, device="cuda")
    f = torch.stack([R.feq(k, one, u) for k in range(19)])
    J = 0.0
    for t in range(T):
        val, gout = R.vibb(f.reshape(19, -1), i, nn, q, ff, ok, torch.zeros_like(arm))
        if t >= T - W:
            J = J - (R.E[i][:, 0] * (gout + val - 2.0 * R.W[i])).sum()
        fin = torch.stack([torch.roll(f[k], (R.e[k][2], R.e[k][1], R.e[k][0]), (0, 1, 2)) for k in range(19)])
        fin = fin.view(19, -1).index_put((i, nn), val).view(19, nz, ny, nx)
        f = torch.stack([torch.where(own < 0, a, b) for a, b in zip(R.collide(fin), f)])
    (J / W).backward()
    return (J / W).item(), scaled(cp.grad.cpu().numpy(), Kt.grad.cpu().numpy())


def test_no_links(pkg):
    """A particle between the nodes: no link, J and the gradient are zero."""
    cp, Kv = np.array([[8.5, 8.5, 8.5]]), np.array([0.1])
    eng = engine(pkg, (16, 17, 18), cp, Kv, 12, 5)
    assert eng.info()["nlinks"] == 0
    assert eng.forward_np(cp, Kv) == 0.0
    g_cp, g_K = eng.backward_np()
    assert not g_cp.any() and not g_K.any()


def test_repeated_calls(pkg):
    """Forward and backward runs repeated on one engine: J to the bit, the
    gradient to the spread of its FP32 atomics (1e-5 of the largest, as in
    tests/test_gpu_adjoint.py)."""
    eng = engine(pkg, (33, 35, 31), CP, K, 40, 10)
    J = eng.forward_np(CP, K)
    g = scaled(*eng.backward_np())
    eng.forward_np(CP + 0.01, K * 1.01)
    eng.backward_np()
    assert eng.forward_np(CP, K) == J
    for _ in range(2):
        assert np.abs(scaled(*eng.backward_np()) - g).max() <= 1e-5 * np.abs(g).max()
