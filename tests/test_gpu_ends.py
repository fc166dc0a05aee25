"""The two ends of a solve: the initial guess read and the solution, norms and flags written by kernels.

Arrays in device memory go through the kernels, host arrays through copies, and the asynchronous solve keeps its norms
on the device; the numbers are the same bit for bit, so every comparison is exact."""
import numpy as np
import pytest

from paper_2206_11294_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n", [(2, 2, 1), (33, 9, 1), (40, 24, 1), (16, 12, 8)])
def test_device_host_and_async_ends_agree(n, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_11294_gb300.binding import Solver
    bc = ((I.BC_WALL, I.BC_DIRICHLET), (I.BC_DIRICHLET, I.BC_WALL), (0, 0))
    g = I.Grid(dim=2 if n[2] == 1 else 3, axisym=0, n=n, h=1e-2, bc=bc, bcT=((300.0, 301.0),) * 3,
               bcp=((1e5, 1.1e5),) * 3)
    p = I.random_coeff_problem(g, seed=sum(n))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    pick = lambda st: [st[k] for k in ("cycles", "r0", "rfinal", "status")]
    with Solver(g, precision=precision, rtol=1e-7, max_cycles=12) as s:
        s.set_coeffs(p.lam, p.fa, p.fk)
        b, x = dev(p.b), dev(p.x0)
        xh, xa = np.array(p.x0, dtype=np.float64, order="C"), dev(p.x0)
        sd = s.solve(b, x, allow_not_converged=True)
        sh = s.solve(p.b, xh, allow_not_converged=True)
        s.solve_async(b, xa)
        sa = s.async_stats(allow_not_converged=True)
        assert np.array_equal(x.cpu().numpy(), xh) and torch.equal(x, xa)
        assert not np.array_equal(xh.reshape(-1), np.asarray(p.x0).reshape(-1))
        assert pick(sd) == pick(sh) == pick(sa)
        r = s.residual_norms(b, xa)
        assert np.array_equal(r, s.residual_norms(p.b, xh)) and torch.equal(x, xa)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("max_cycles,rtol", [(0, 1e-7), (1, 1e-7), (12, 1e-7), (12, 1.0), (3, 0.0)])
def test_batch_ends_agree(max_cycles, rtol, precision):
    """The first cycle runs ahead of the initial norms: problems that met the test at the start are left as they were."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_11294_gb300.binding import Batch, Solver
    bc = ((I.BC_WALL, I.BC_DIRICHLET), (I.BC_DIRICHLET, I.BC_WALL), (0, 0))
    problems = [I.random_coeff_problem(I.Grid(dim=2, axisym=0, n=n, h=1e-2, bc=bc, bcT=((300.0, 301.0),) * 3,
                                              bcp=((1e5, 1.1e5),) * 3), seed=sum(n))
                for n in ((33, 9, 1), (40, 24, 1), (8, 4, 1))]
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    solvers = [Solver(p.grid, precision=precision, rtol=rtol, max_cycles=max_cycles) for p in problems]
    batch = Batch(solvers)
    batch.set_coeffs([p.lam for p in problems], [p.fa for p in problems], [p.fk for p in problems])
    xd, xh = [dev(p.x0) for p in problems], [np.array(p.x0, order="C") for p in problems]
    sd = batch.solve([dev(p.b) for p in problems], xd, allow_not_converged=True)
    sh = batch.solve([p.b for p in problems], xh, allow_not_converged=True)
    for p, a, h, d, e in zip(problems, xd, xh, sd, sh):
        assert np.array_equal(a.cpu().numpy(), h)
        assert [d[k] for k in ("cycles", "r0", "rfinal")] == [e[k] for k in ("cycles", "r0", "rfinal")]
        want = 0 if max_cycles == 0 or rtol >= 1.0 else max_cycles if rtol <= 0.0 else None
        assert want is None or d["outer"] == want, d
        assert (d["outer"] > 0) == (not np.array_equal(h.reshape(-1), np.asarray(p.x0).reshape(-1)))
    batch.close()
    for s in solvers:
        s.close()


def test_arrays_of_the_wrong_kind_are_refused_as_before():
    """One look at plain CUDA tensors; anything else goes the general way and raises there."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_11294_gb300.binding import Batch, Solver
    g = I.Grid(dim=2, axisym=0, n=(8, 4, 1), h=1e-2, bc=((I.BC_WALL, I.BC_WALL),) * 2 + ((0, 0),))
    p = I.random_coeff_problem(g, seed=3)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    s = Solver(g, rtol=0.0, max_cycles=1)
    batch = Batch([s])
    lam, fa, fk, b, x = dev(p.lam), [dev(f) for f in p.fa], [dev(f) for f in p.fk], dev(p.b), dev(p.x0)
    wide = torch.zeros(2 * b.numel(), dtype=torch.float64, device="cuda")
    for bad, error in ((b.reshape(-1)[:-2], ValueError), (b.float(), TypeError), (wide[::2], TypeError),
                       (b.cpu(), TypeError)):
        s.set_coeffs(lam, fa, fk)
        for call in (lambda: s.solve(bad, x), lambda: batch.solve([bad], [x])):
            with pytest.raises(error):
                call()
    for bad, error in ((fa[:1], (ValueError, IndexError)), ([fa[0], fa[0][:-1]], ValueError), ([fa[0], fa[1].cpu()], TypeError)):
        for call in (lambda: s.set_coeffs(lam, bad, fk), lambda: batch.set_coeffs([lam], [bad], [fk])):
            with pytest.raises(error):
                call()
    s.set_coeffs(lam, fa + [fa[0]], fk)          # more face arrays than axes: the first ones count
    st = s.solve(b, x)
    assert st["cycles"] == 1
    batch.close()
    s.close()
