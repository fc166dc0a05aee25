"""The coarsest solve alone: grids that are their own coarsest level.

One cycle of such a grid is the exact solve, so the result is compared with
the dense solution.  Sizes: inverses up to 128 unknowns and block cyclic
reduction above, blocks along each axis, block counts around powers of two, the
largest grid, 3D blocks.  The fallback (banded LU with partial pivoting) runs
where a 2 x 2 pivot block is exactly singular while the matrix is not.

Tolerances: a solve's forward error is at most cond * eps * growth; the block
rows dominate in these problems (cond of the row-scaled matrix below 1e3), so
1e-12 of the solution for FP64; mixed precision converges to the FP64
right-hand side's solution at 1e-10, checked at 1e-8 as elsewhere.
"""
import numpy as np
import pytest

from paper_2206_11294_gb300 import inputs as I
from tests.fv_matrix import paper_operator

pytestmark = pytest.mark.gpu
W, D = I.BC_WALL, I.BC_DIRICHLET

SHAPES = [(4, 4, 1), (5, 7, 1), (7, 9, 1), (9, 13, 1), (13, 9, 1), (29, 4, 1), (4, 29, 1), (15, 15, 1), (31, 31, 1),
          (4, 4, 4), (5, 5, 5), (7, 6, 7), (6, 8, 10), (3, 2, 33)]


@pytest.fixture(scope="module")
def binding():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_11294_gb300 import binding as b
    b.load()
    return b


def _grid(n):
    dim = 2 if n[2] == 1 else 3
    bc = ((W, D), (D, W), (W, W)) if dim == 3 else ((W, D), (W, W), (0, 0))
    return I.Grid(dim=dim, axisym=0, n=n, h=1e-2, bc=bc, bcT=((300.0, 300.0),) * 3, bcp=((1e5, 1e5),) * 3)


def _rel(x, ref, x0):
    return max(np.linalg.norm(x[:, f] - ref[:, f]) / np.linalg.norm(ref[:, f] - x0[:, f]) for f in range(2))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n", SHAPES, ids=lambda n: "x".join(map(str, n)))
def test_single_level_solve_is_the_dense_solution(binding, n, precision):
    import oracle
    p = I.random_coeff_problem(_grid(n), seed=sum(n))
    ref = oracle.dense_solve(p.grid.as_dict(), p.lam, p.fa, p.fk, p.b)
    kw = dict(rtol=0.0, max_cycles=1) if precision == "fp64" else dict(rtol=1e-10, max_cycles=20)
    s = binding.Solver(p.grid, precision=precision, **kw)
    assert len(s.levels()) == 1
    s.set_coeffs(p.lam, p.fa, p.fk)
    x = p.x0.copy()
    s.solve(p.b, x)
    assert _rel(x, ref, p.x0) <= (1e-12 if precision == "fp64" else 1e-8)
    s.close()


def _singular_pivot(n):
    """Unit faces; the first cell's block and the second's after its elimination are [1, 0; 0, .] and [0, 0; 0, .]."""
    g = I.Grid(dim=2, axisym=0, n=n, h=1.0, bc=((W, W), (W, W), (0, 0)))
    lam = np.zeros((g.N, 4))
    lam[:, 0] = lam[:, 2] = -10.0
    lam[0, 0], lam[1, 0] = 1.0 + 2.0, 1.0 + 3.0          # minus the 2 and 3 interior faces of the two cells
    ones = [np.ones(g.face_shape(a)).reshape(-1) for a in range(2)]
    return g, lam, ones


@pytest.mark.parametrize("n", [(7, 7, 1), (9, 13, 1)], ids=["inverse", "reduction"])
def test_singular_pivot_block_takes_the_pivoted_factors(binding, n):
    g, lam, ones = _singular_pivot(n)
    A = paper_operator(g, lam, ones, ones)
    A = np.asarray((A[0] if isinstance(A, tuple) else A).todense())
    rng = np.random.default_rng(3)
    xs = rng.normal(size=(g.N, 2))
    b = (A @ xs.reshape(-1)).reshape(-1, 2)
    for batched in (False, True):
        solvers = [binding.Solver(g, rtol=0.0, max_cycles=1) for _ in range(2 if batched else 1)]
        x = np.zeros((g.N, 2))
        if batched:
            batch = binding.Batch(solvers)
            batch.set_coeffs([lam] * 2, [ones] * 2, [ones] * 2)
            batch.solve([b] * 2, [x, np.zeros_like(x)])
            batch.close()
        else:
            solvers[0].set_coeffs(lam, ones, ones)
            solvers[0].solve(b, x)
        # cond(A) bounds the error of a backward stable solve
        assert np.abs(x - xs).max() <= 16 * np.finfo(float).eps * np.linalg.cond(A) * np.abs(xs).max()
        for s in solvers:
            s.close()


def test_singular_matrix_is_still_refused(binding):
    g, lam, ones = _singular_pivot((9, 13, 1))
    k = [f.reshape(g.face_shape(a)).copy() for a, f in enumerate(ones)]
    k[0][0, 0, 2] = k[1][0, 1, 0] = k[1][0, 1, 1] = 0.0   # the first two cells' T coupled to each other only,
    lam[0, 0] = lam[1, 0] = 2.0                           # with equal rows [1, 1]
    fk = [f.reshape(-1) for f in k]
    for batched in (False, True):
        s = binding.Solver(g, rtol=0.0, max_cycles=1)
        with pytest.raises(Exception, match="singular"):
            if batched:
                binding.Batch([s]).set_coeffs([lam], [ones], [fk])
            else:
                s.set_coeffs(lam, ones, fk)
                s.solve(np.zeros((g.N, 2)), np.zeros((g.N, 2)))
        s.close()


@pytest.mark.parametrize("delta", [1e-2, 1e-4, 1e-6, 1e-8, 1e-10, 1e-12, 1e-14])
@pytest.mark.parametrize("n", [(7, 7, 1), (9, 13, 1)], ids=["inverse", "reduction"])
def test_nearly_singular_pivot_block(binding, n, delta):
    """The second pivot block after the first one's elimination is delta away from singular: elimination without row
    exchanges loses a factor 1 / delta.  A grid that is its own coarsest level is solved from these factors alone, so
    its error stays within the bound of a backward stable solve, 16 eps cond(A) (test above)."""
    g, lam, ones = _singular_pivot(n)
    lam[1, 0] += delta
    A = paper_operator(g, lam, ones, ones)
    A = np.asarray((A[0] if isinstance(A, tuple) else A).todense())
    xs = np.random.default_rng(3).normal(size=(g.N, 2))
    b = (A @ xs.reshape(-1)).reshape(-1, 2)
    for batched in (False, True):
        s = binding.Solver(g, rtol=0.0, max_cycles=1)
        x = np.zeros((g.N, 2))
        if batched:
            batch = binding.Batch([s])
            batch.set_coeffs([lam], [ones], [ones])
            batch.solve([b], [x])
            batch.close()
        else:
            s.set_coeffs(lam, ones, ones)
            s.solve(b, x)
        s.close()
        assert np.abs(x - xs).max() <= 16 * np.finfo(float).eps * np.linalg.cond(A) * np.abs(xs).max()


def test_long_thin_coarsest_grid(binding):
    """300 blocks of 4 unknowns: nine elimination stages."""
    test_single_level_solve_is_the_dense_solution(binding, (2, 300, 1), "fp64")


def test_blocks_above_the_inverse_beside_smaller_ones(binding):
    """9 x 9 x 9 cells have blocks of 162 unknowns, too large for the cluster inverse (kGjMax): in a batch they keep the
    banded LU while 5 x 5 x 5 and 7 x 6 x 7 take the reduction."""
    import oracle
    probs = [I.random_coeff_problem(_grid(n), seed=sum(n)) for n in ((5, 5, 5), (9, 9, 9), (7, 6, 7))]
    solvers = [binding.Solver(p.grid, rtol=0.0, max_cycles=1) for p in probs]
    batch = binding.Batch(solvers)
    batch.set_coeffs([p.lam for p in probs], [p.fa for p in probs], [p.fk for p in probs])
    xs = [p.x0.copy() for p in probs]
    batch.solve([p.b for p in probs], xs)
    for p, x in zip(probs, xs):
        ref = oracle.dense_solve(p.grid.as_dict(), p.lam, p.fa, p.fk, p.b)
        assert _rel(x, ref, p.x0) <= 1e-12, p.grid.n
    batch.close()
    for s in solvers:
        s.close()


@pytest.mark.parametrize("n", [(1, 90, 1), (2, 40, 1), (3, 50, 1), (2, 300, 1)], ids=lambda n: "x".join(map(str, n)))
def test_banded_factors_of_narrow_grids(binding, n):
    """Bands narrower than a panel of the blocked LU (three columns and less along the fast axis), by the inverse it
    forms and, with a nearly singular pivot block, as the reduction's fallback.  The tolerances are the ones above."""
    import oracle
    p = I.random_coeff_problem(_grid(n), seed=sum(n))
    ref = oracle.dense_solve(p.grid.as_dict(), p.lam, p.fa, p.fk, p.b)
    s = binding.Solver(p.grid, rtol=0.0, max_cycles=1, coarse="inverse")
    assert len(s.levels()) == 1
    s.set_coeffs(p.lam, p.fa, p.fk)
    x = p.x0.copy()
    s.solve(p.b, x)
    s.close()
    assert _rel(x, ref, p.x0) <= 1e-12
    g, lam, ones = _singular_pivot(n)
    if n[0] < 3:
        lam[0, 0], lam[1, 0] = 1.0 + n[0], 1.0 + 2.0         # one or two interior faces, and two
    A = paper_operator(g, lam, ones, ones)
    A = np.asarray((A[0] if isinstance(A, tuple) else A).todense())
    xs = np.random.default_rng(3).normal(size=(g.N, 2))
    b = (A @ xs.reshape(-1)).reshape(-1, 2)
    x = np.zeros((g.N, 2))
    s = binding.Solver(g, rtol=0.0, max_cycles=1)
    s.set_coeffs(lam, ones, ones)
    s.solve(b, x)
    s.close()
    assert np.abs(x - xs).max() <= 16 * np.finfo(float).eps * np.linalg.cond(A) * np.abs(xs).max()
