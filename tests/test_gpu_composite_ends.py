"""The copies either side of a refined-patch solve, and its first sweeps from zero.

Coefficients in arrays aligned to 8 bytes only and the same in aligned ones (of odd lengths too) give the same solution
bit for bit.  Without sweeps before the base correction (nu1 = 0) the patch's correction starts from a
cleared array; with them the first colour must not read it: either way three cycles from zero at least halve the residual
(an unsound start leaves it where it was or worse; a sound cycle takes several times that)."""
import numpy as np
import pytest

from paper_2206_11294_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _dev(torch, a, shift=0):
    a = np.ascontiguousarray(a, dtype=np.float64).reshape(-1)
    t = torch.zeros(a.size + 2, dtype=torch.float64, device="cuda")[shift:shift + a.size]
    t.copy_(torch.from_numpy(a).cuda())
    return t


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.parametrize("n,box", [((16, 9), ((3, 9), (2, 6))), ((21, 21), ((20, 21), (0, 21))), ((40, 24), ((1, 39), (4, 5)))])
def test_copies_of_any_alignment(torch_cuda, n, box):
    from paper_2206_11294_gb300.binding import Composite
    bc = ((I.BC_WALL, I.BC_DIRICHLET), (I.BC_DIRICHLET, I.BC_WALL), (0, 0))
    grid = lambda m, h: I.Grid(dim=2, axisym=0, n=m + (1,), h=h, bc=bc, bcT=((300.0, 301.0),) * 3,
                               bcp=((1e5, 1.1e5),) * 3)
    b = I.random_coeff_problem(grid(n, 1e-2), seed=1)
    p = I.random_coeff_problem(grid(tuple(2 * (q[1] - q[0]) for q in box), 5e-3), seed=2)
    out = []
    for shift in (0, 1):
        c = Composite(b.grid, box)
        d = lambda a: _dev(torch_cuda, a, shift)
        c.set_coeffs(d(b.lam), [d(f) for f in b.fa], [d(f) for f in b.fk], d(p.lam), [d(f) for f in p.fa],
                     [d(f) for f in p.fk])
        v = [_dev(torch_cuda, a) for a in (b.b, p.b, b.x0, p.x0)]
        c.solve(*v, cycles=2, norms=False)
        out.append([a.cpu().numpy() for a in v[2:]])
        c.close()
    assert all(np.isfinite(a).all() and np.array_equal(a, e) for a, e in zip(*out))


@pytest.mark.parametrize("nu1,nu2", [(0, 2), (1, 1), (2, 0)])
def test_first_sweep_from_zero(torch_cuda, nu1, nu2):
    from paper_2206_11294_gb300.binding import Composite
    b, p, box = I.composite_bubble(48, box=((0, 20), (0, 24)), seed=23, n_bubbles=1, rmin=0.08, rmax=0.12)
    c = Composite(b.grid, box, nu1=nu1, nu2=nu2)
    c.set_coeffs(b.lam, b.fa, b.fk, p.lam, p.fa, p.fk)
    x = [0.0 * _dev(torch_cuda, a) for a in (b.x0, p.x0)]
    norms = c.solve(_dev(torch_cuda, b.b), _dev(torch_cuda, p.b), *x, cycles=3)[2]
    for f in range(2):
        total = np.hypot(norms[:, f], norms[:, 2 + f])
        assert np.isfinite(total).all() and total[3] <= 0.5 * total[0], (nu1, nu2, total)
    c.close()


@pytest.mark.parametrize("cycles", [1, 2])
@pytest.mark.parametrize("nu1,nu2", [(0, 2), (1, 1), (2, 0), (3, 1)])
def test_sweep_counts_match_the_oracle(torch_cuda, nu1, nu2, cycles):
    """The cycle from a cleared correction (nu1 = 0), from its first colour, and without post-sweeps, within 1e-12 of the
    oracle's in the deviation from the guess (the tolerance of the default counts)."""
    from oracle import composite as cf
    from paper_2206_11294_gb300.binding import Composite
    b, p, box = I.composite_bubble(48, box=((0, 20), (0, 24)), seed=23, n_bubbles=1, rmin=0.08, rmax=0.12)
    c = Composite(b.grid, box, nu1=nu1, nu2=nu2)
    c.set_coeffs(b.lam, b.fa, b.fk, p.lam, p.fa, p.fk)
    x = [_dev(torch_cuda, a) for a in (b.x0, p.x0)]
    c.solve(_dev(torch_cuda, b.b), _dev(torch_cuda, p.b), *x, cycles=cycles, norms=False)
    ref = cf.fac_solve(b.grid.as_dict(), box, b.lam, b.fa, b.fk, p.lam, p.fa, p.fk, b.b, p.b, b.x0, p.x0, cycles, nu1=nu1,
                       nu2=nu2)
    for got, want, start in zip(x, ref, (b.x0, p.x0)):
        got = got.cpu().numpy().reshape(-1, 2)
        for f in range(2):
            assert np.abs(got[:, f] - want[:, f]).max() <= 1e-12 * np.abs(want[:, f] - start[:, f]).max()
    c.close()
