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
