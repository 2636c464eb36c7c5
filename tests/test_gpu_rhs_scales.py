"""GPU: right-hand sides of very different sizes in one hierarchy.

The copies of the grid that carry the right-hand sides are independent: the sweeps on two of
them give what a single-right-hand-side hierarchy gives for each, to the 1e-11 of the other
FP64 parity tests (the two differ by the order of the atomic additions, at most eight per
node, 1e-15 each), however far apart the two are.
"""
import numpy as np
import pytest

import synthetic as syn
from tests.helpers import elem_shape, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GRIDS = [(3, 4, [[0.3, 0.5, 0.2], [0.6, 0.4], [0.7, 0.3]]), (3, 8, [[0.5, 0.5], [0.3, 0.7], [0.25] * 4]),
         (3, 16, [[1.0], [0.4, 0.6], [0.5, 0.5]]), (2, 8, [[0.3, 0.5, 0.2], [0.4, 0.1, 0.5]])]


@pytest.mark.parametrize("k", [40, -40, 70, -70])
@pytest.mark.parametrize("kind", ["EA", "FA"])
@pytest.mark.parametrize("dim,P,sp", GRIDS, ids=[f"{g[0]}d-P{g[1]}" for g in GRIDS])
def test_sweeps_of_unlike_right_hand_sides(dim, P, sp, kind, k):
    from paper_1603_02524_gb300 import Grid, Hierarchy
    ne = [len(s) for s in sp]
    g = Grid(dim, P, ne, sp, periodic=False)
    h1, h2 = Hierarchy(g, smoother=kind), Hierarchy(g, smoother=kind, nrhs=2)
    r = [to_dev(syn.rng(120 + i).uniform(-1, 1, size=elem_shape(dim, ne, P))) for i in range(2)]
    r[1] = r[1] * 2.0 ** k
    for fam in [-1] if kind == "EA" else range(dim):
        both = torch.zeros(2 * h1.ndof(), dtype=torch.float64, device="cuda")
        h2.schwarz_sweep(h2.L, fam, torch.cat(r), both)
        for i in range(2):
            one = torch.zeros_like(r[i])
            h1.schwarz_sweep(h1.L, fam, r[i], one)
            diff = (both[i * one.numel():(i + 1) * one.numel()] - one).abs().max()
            assert float(diff) <= 1e-11 * float(one.abs().max())
