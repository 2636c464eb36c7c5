"""GPU: the exact coarse solve on lines longer than the staged kernel takes (2048 coarse nodes).

Right-hand sides are stacked along the last axis, so 17 elements and 64 of them make 2176 coarse
nodes.  Each right-hand side's solution is that of a hierarchy of its own: 1e-12, the coarse
solve's parity tolerance (sums of at most 34 nonzero products, eigenvectors from the same Jacobi
rotations in another order).
"""
import pytest

import synthetic as syn
from tests.helpers import elem_shape, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("ne", [(3, 17), (2, 3, 17)])
def test_coarse_solve_of_long_lines(ne, precision):
    from paper_1603_02524_gb300 import Grid, Hierarchy
    dim, K = len(ne), 64
    sp = [[1.0 / n] * n for n in ne]
    g = Grid(dim, 2, ne, sp, periodic=False)
    h1, hk = Hierarchy(g, precision=precision), Hierarchy(g, nrhs=K, precision=precision)
    n = h1.ndof(0)
    f = to_dev(syn.rng(170).uniform(-1, 1, size=(K,) + elem_shape(dim, ne, 1)))
    u = torch.empty_like(f)
    hk.coarse_solve(f, u)
    for i in (0, 1, 31, K - 1):
        one = torch.empty(n, dtype=torch.float64, device="cuda")
        h1.coarse_solve(f[i * n:(i + 1) * n], one)
        assert float((u[i * n:(i + 1) * n] - one).abs().max()) <= 1e-12 * float(one.abs().max())
    # and inside a V-cycle (fp32 vectors in the mixed one)
    m = h1.ndof()
    r = to_dev(syn.rng(171).uniform(-1, 1, size=(K,) + elem_shape(dim, ne, 2)))
    z = torch.empty_like(r)
    hk.vcycle(r, z)
    one = torch.empty(m, dtype=torch.float64, device="cuda")
    h1.vcycle(r[:m].contiguous(), one)
    tol = 1e-10 if precision == "fp64" else 1e-5
    assert float((z[:m] - one).abs().max()) <= tol * float(one.abs().max())
