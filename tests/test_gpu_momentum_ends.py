"""The point-Jacobi loop's device-side ends: the first step sets the correction, the last adds it to the velocity, and
a start that meets the test, no step allowed or a residual that is not finite leave the velocity as it was.

Two steps in one call against two calls of one step: both form the same corrections, the second from r0 - A(delta) or
from R - A(u).  A row of R - A(u) rounds within about ten units of rho u / dt (the viscous terms are 1e-3 of it here),
which the diagonal turns into ten units of u; 64 eps max|u| leaves room for both calls' updates."""
import numpy as np
import pytest

from paper_2206_11294_gb300 import inputs as I

pytestmark = pytest.mark.gpu

W, D = I.BC_WALL, I.BC_DIRICHLET


@pytest.mark.parametrize("n", [(33, 9, 1), (40, 36, 1), (12, 10, 8)])
def test_jacobi_loop_ends(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_11294_gb300.binding import MgError, Momentum
    dim = 2 if n[2] == 1 else 3
    g = I.Grid(dim=dim, axisym=0, n=n, h=1e-2, bc=((W, D), (W, W), (D, W) if dim == 3 else (0, 0)))
    rng = np.random.default_rng(sum(n))
    shape = (n[2], n[1], n[0])
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()
    rho, mu, dt = rng.uniform(1.0, 1000.0, shape), 1e-4 * rng.uniform(1e-3, 1.0, shape), 1e-4
    u0 = [rng.normal(size=shape) for _ in range(dim)]
    R = [dev(rho / dt * (v + 0.1 * rng.normal(size=shape))) for v in u0]
    m = Momentum(g)
    m.set_coeffs(dt, dev(rho), dev(mu))

    def steps(*counts, rhs=R, rtol=0.0):
        u = [dev(v) for v in u0]
        st = [m.solve(rhs, u, rtol=rtol, max_iters=k, allow_not_converged=True) for k in counts]
        return [v.cpu().numpy() for v in u], st

    one, st = steps(2)
    two, st2 = steps(1, 1)
    assert st[0]["jacobi"] and st[0]["iterations"] == 2 and st2[1]["iterations"] == 1
    top = max(np.abs(v).max() for v in one)
    for a, b, v in zip(one, two, u0):
        assert np.abs(a - b).max() <= 64 * np.finfo(float).eps * top and np.abs(a - v).max() > 1e-3
    for kw, count in ((dict(), 0), (dict(rtol=1.0), 5)):
        same, st = steps(count, **kw)
        assert st[0]["iterations"] == 0 and all(np.array_equal(a, v) for a, v in zip(same, u0))
    bad = [r.clone() for r in R]
    bad[0].view(-1)[7] = float("nan")
    u = [dev(v) for v in u0]
    with pytest.raises(MgError):
        m.solve(bad, u, rtol=1e-8, max_iters=3)
    assert all(np.array_equal(a.cpu().numpy(), v) for a, v in zip(u, u0))
    m.close()


def _nan(negative):
    return np.array([0xFFF8000000000000 if negative else 0x7FF8000000000000], dtype=np.uint64).view(np.float64)[0]


@pytest.mark.parametrize("grid", ["2d", "axi", "3d"])
def test_coefficients_that_are_not_finite(grid):
    """One NaN of either sign in rho or mu, or an infinite mu, among cells whose row bound is far below the limit of the
    point-Jacobi corrections: the set-up reports it, from an inner cell and from one at the boundary."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_11294_gb300.binding import MG_ERR_INVALID_COEFF, MgError, Momentum
    n = (12, 10, 8) if grid == "3d" else (40, 36, 1)
    bc = ((I.BC_AXIS if grid == "axi" else W, D), (W, W), (D, W) if grid == "3d" else (0, 0))
    g = I.Grid(dim=3 if grid == "3d" else 2, axisym=int(grid == "axi"), n=n, h=1e-2, bc=bc)
    rng = np.random.default_rng(5)
    shape = (n[2], n[1], n[0])
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()
    rho, mu, dt = rng.uniform(1.0, 1000.0, shape), 1e-4 * rng.uniform(1e-3, 1.0, shape), 1e-4
    m = Momentum(g)
    for field, value in (("rho", _nan(False)), ("rho", _nan(True)), ("mu", _nan(False)), ("mu", _nan(True)),
                         ("mu", np.inf)):
        for cell in ((n[2] // 2, 5, 7), (0, 0, n[0] - 1)):
            f = dict(rho=rho.copy(), mu=mu.copy())
            f[field][cell] = value
            with pytest.raises(MgError) as e:
                m.set_coeffs(dt, dev(f["rho"]), dev(f["mu"]))
            assert e.value.status == MG_ERR_INVALID_COEFF, (field, value, cell)
    m.set_coeffs(dt, dev(rho), dev(mu))
    m.close()
