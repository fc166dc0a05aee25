"""Coefficient intake: lambda aligned to 8 bytes only, and the jump marks of the integer comparison.

Both are exact: the same numbers must give the same solution bit for bit, and the number of marked cells is an
integer that numpy counts from the face arrays (with values of either sign and zeros)."""
import numpy as np
import pytest

from paper_2206_11294_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_11294_gb300 import binding
    binding.load()
    return torch


def _problem(n, axisym=0):
    dim = 2 if n[2] == 1 else 3
    bc = ((I.BC_WALL, I.BC_DIRICHLET), (I.BC_DIRICHLET, I.BC_WALL), (0, 0))
    if axisym:
        bc = ((I.BC_AXIS, I.BC_DIRICHLET),) + bc[1:]
    g = I.Grid(dim=dim, axisym=axisym, n=n, h=1e-2, bc=bc, bcT=((300.0, 301.0),) * 3, bcp=((1e5, 1.1e5),) * 3)
    return I.random_coeff_problem(g, seed=sum(n))


@pytest.mark.parametrize("n,axisym", [((40, 24, 1), 0), ((40, 24, 1), 1), ((33, 9, 1), 0), ((16, 12, 8), 0)])
def test_lambda_aligned_to_8_bytes(torch_cuda, n, axisym):
    torch = torch_cuda
    from paper_2206_11294_gb300.binding import Solver
    p = _problem(n, axisym)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    out = []
    for shift in (0, 1):
        buf = torch.zeros(p.lam.size + 2, dtype=torch.float64, device="cuda")
        lam = buf[shift:shift + p.lam.size]
        lam.copy_(dev(p.lam.reshape(-1)))
        assert lam.data_ptr() % 16 == 8 * shift
        s = Solver(p.grid, rtol=0.0, max_cycles=2)
        s.set_coeffs(lam, [dev(f) for f in p.fa], [dev(f) for f in p.fk])
        x = dev(p.x0)
        s.solve(dev(p.b), x)
        out.append(x.cpu().numpy())
        s.close()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("n", [(40, 24, 1), (33, 9, 1), (16, 12, 8)])
def test_jump_marks_with_values_of_either_sign(torch_cuda, n):
    from paper_2206_11294_gb300.binding import Solver
    p = _problem(n)
    rng = np.random.default_rng(1)
    fk = [f * rng.choice([1.0, 1.0, 1.0, -1.0, 0.0], size=f.shape) * rng.uniform(0.6, 1.6, f.shape) for f in p.fk]
    s = Solver(p.grid, precision="mixed", rtol=0.0, max_cycles=1, fp64_jump_ratio=2.0)
    s.set_coeffs(p.lam, p.fa, fk)
    got = s.solve(p.b, p.x0.copy())["fp64_cells"]
    s.close()
    g, shape = p.grid, (n[2], n[1], n[0])
    marked = np.zeros(shape, dtype=bool)
    for faces in (p.fa, fk):
        lo, hi = np.full(shape, np.inf), np.full(shape, -np.inf)
        for a in range(g.dim):
            f = faces[a].reshape(g.face_shape(a))
            low, high = np.take(f, range(n[a]), 2 - a).copy(), np.take(f, range(1, n[a] + 1), 2 - a).copy()
            first = [slice(None)] * 3
            last = [slice(None)] * 3
            first[2 - a], last[2 - a] = slice(0, 1), slice(-1, None)
            for v, edge in ((low, first), (high, last)):
                inner = np.ones(shape, dtype=bool)
                inner[tuple(edge)] = False                 # boundary faces do not count
                lo = np.where(inner, np.minimum(lo, v), lo)
                hi = np.where(inner, np.maximum(hi, v), hi)
        marked |= hi > 2.0 * lo
    assert got == int(marked.sum())
