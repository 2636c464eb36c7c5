"""GPU: the digit-split FP64 kernels keep FP64 precision where values of very different size meet.

Every bound is relative to what a value is formed from, not to the largest value around it.
"""
import numpy as np
import pytest

import synthetic as syn
from oracle import dg, schwarz
from tests.helpers import e2g, elem_shape, from_dev, g2e, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fam", [0, 1, 2])
@pytest.mark.parametrize("P,overlap", [(8, "l"), (16, "0"), (16, "l")])
def test_sweep_precision_under_small_weights(P, overlap, fam):
    """A residual in the first of three elements along the normal: the second one's nodes take
    their corrections from one face patch, whose weights fall to about 1e-6 of the largest.
    Every plane of nodes agrees with the oracle to the sweeps' 1e-11 of that plane's largest."""
    from paper_1603_02524_gb300 import Grid, Hierarchy
    sp = [[1.0], [0.7], [0.8]]
    sp[fam] = [1 / 3] * 3
    ne = [len(s) for s in sp]
    shape = elem_shape(3, ne, P)
    r = np.zeros(shape)
    r[0, 0, 0] = syn.rng(130 + P).uniform(-1, 1, size=shape[3:])
    h = Hierarchy(Grid(3, P, ne, sp, periodic=False), smoother="FA", overlap=overlap)
    out = torch.zeros(r.size, dtype=torch.float64, device="cuda")
    h.schwarz_sweep(h.L, fam, to_dev(r), out)
    sm = schwarz.Smoother(dg.Discretisation(3, P, sp, False, 0.0, 1.0), "FA", overlap, "quintic")
    ref = np.moveaxis(sm.additive_sweep(np.zeros_like(e2g(r, 3)), e2g(r, 3), normal=fam), 2 - fam, 0)
    got = np.moveaxis(e2g(from_dev(out, shape), 3), 2 - fam, 0)
    for k in range(2 * P + 1):
        assert np.abs(got[k] - ref[k]).max() <= 1e-11 * np.abs(ref[k]).max()


GRID = [[0.25] * 4, [0.5] * 2, [0.3, 0.7]]


@pytest.mark.parametrize("big", [1e12, 1e30, -1e250])
@pytest.mark.parametrize("P", [4, 8, 16])
def test_apply_off_the_lines_of_a_large_value(P, big):
    """A u depends on the lines through a node: one large value changes nothing elsewhere."""
    from paper_1603_02524_gb300 import Grid, Hierarchy
    h = Hierarchy(Grid(3, P, [4, 2, 2], GRID, periodic=False))
    shape = elem_shape(3, (4, 2, 2), P)
    u = syn.rng(140).uniform(-1, 1, size=shape)
    a, b = (torch.zeros(u.size, dtype=torch.float64, device="cuda") for _ in range(2))
    h.apply(h.L, to_dev(u), a)
    u[0, 0, 1, 1, 2, 2] = big
    h.apply(h.L, to_dev(u), b)
    hit = np.zeros(shape, dtype=bool)
    hit[0, 0, :3, 1, 2, :] = hit[0, 0, 1, 1, :, 2] = hit[0, 0, 1, :, 2, 2] = True
    hit[0, 1, 1, 1, :, 2] = hit[1, 0, 1, :, 2, 2] = True
    got, ref = from_dev(b, shape), from_dev(a, shape)
    assert np.abs(got[~hit] - ref[~hit]).max() <= 1e-13 * np.abs(ref).max()


@pytest.mark.parametrize("small", [1e-6, 1e-15, 1e-290])
@pytest.mark.parametrize("P", [4, 8, 16])
def test_apply_at_small_edges(P, small):
    """Values far smaller on two faces of every element (as next to a Dirichlet wall): the edge
    between them depends on these alone and keeps the relative accuracy of the apply."""
    from paper_1603_02524_gb300 import Grid, Hierarchy
    h = Hierarchy(Grid(3, P, [4, 2, 2], GRID, periodic=False))
    shape = elem_shape(3, (4, 2, 2), P)
    u = syn.rng(141).uniform(-1, 1, size=shape)
    u[..., 0, :] *= small
    u[..., 0] *= small
    u[..., 0, 0] /= small
    out = torch.zeros(u.size, dtype=torch.float64, device="cuda")
    h.apply(h.L, to_dev(u), out)
    v = u.copy()                                           # the rest zero: the edge's result is the same
    v[..., 1:, 1:] = 0.0
    v /= small
    ref = g2e(dg.Discretisation(3, P, GRID, False, 0.0, 1.0).apply(e2g(v, 3)), (4, 2, 2), P)[..., 0, 0]
    got = from_dev(out, shape)[..., 0, 0] / small
    assert np.abs(got - ref).max() <= 1e-13 * np.abs(ref).max()


@pytest.mark.parametrize("P", [4, 8, 16])
def test_apply_of_a_localized_vector(P):
    """Zero but for one element: the other elements' results are exact zeros, and they take no
    longer than full ones (twice the time is the bound)."""
    from paper_1603_02524_gb300 import Grid, Hierarchy
    ne = (8, 8, 8)
    sp = [[1 / n] * n for n in ne]
    h = Hierarchy(Grid(3, P, ne, sp, periodic=False))
    shape = elem_shape(3, ne, P)
    u = np.zeros(shape)
    u[4, 3, 2] = syn.rng(142).uniform(-1, 1, size=shape[3:])
    full = torch.rand(u.size, dtype=torch.float64, device="cuda")
    loc, out = to_dev(u), torch.empty_like(full)
    h.apply(h.L, loc, out)
    got = from_dev(out, shape)
    near = np.zeros(shape[:3], dtype=bool)
    near[4, 3, 1:4] = near[4, 2:5, 2] = near[3:6, 3, 2] = True
    assert (got[~near] == 0.0).all() and (got[near] != 0.0).any()

    def ms(x):
        best = 1e9
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                h.apply(h.L, x, out)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best
    assert ms(loc) <= 2.0 * ms(full)


@pytest.mark.parametrize("P", [4, 8, 16])
def test_apply_errors_have_no_sign(P):
    """A u + A (-u) is the sum of two rounding errors.  Where they are of one sign all over a field,
    coarse grids and smoothers add them up; of N random signs the surplus is about sqrt(N), far
    below a tenth of the 2000 to 90 000 nodes here."""
    from paper_1603_02524_gb300 import Grid, Hierarchy
    sp = [[1 / 3] * 3, [0.3, 0.5, 0.2], [0.6, 0.4]]
    h = Hierarchy(Grid(3, P, [3, 3, 2], sp, periodic=False))
    u = to_dev(syn.rng(160).uniform(-1, 1, size=elem_shape(3, (3, 3, 2), P)))
    a, b = torch.empty_like(u), torch.empty_like(u)
    h.apply(h.L, u, a)
    h.apply(h.L, -u, b)
    s = a + b
    assert abs(int((s > 0).sum()) - int((s < 0).sum())) <= 0.1 * u.numel()


@pytest.mark.parametrize("P", [4, 8, 16])
def test_prolongation_keeps_small_values(P):
    """A face of a fine element depends on that face of the coarse one alone, and values of 1e-9 to
    1 keep their relative accuracy on the lines they are formed from (1e-13, as the transfers'
    parity tests; a line's values enter in mirrored pairs)."""
    from oracle.mg import Hierarchy as OHier
    from paper_1603_02524_gb300 import Grid, Hierarchy
    h, oh = Hierarchy(Grid(3, P, [4, 2, 2], GRID, periodic=False)), OHier(3, P, GRID, False)
    sc, sf = elem_shape(3, (4, 2, 2), P // 2), elem_shape(3, (4, 2, 2), P)
    c = syn.rng(150).uniform(-1, 1, size=sc)
    c[..., 1:-1, 1:-1, 1:-1] *= 1e20                           # off the faces
    c[..., 0] *= 1e-9                                          # two small faces
    c[..., -1] *= 1e-9
    out = torch.zeros(int(np.prod(sf)), dtype=torch.float64, device="cuda")
    h.prolong(h.L, to_dev(c), out)
    got, ref = from_dev(out, sf), g2e(oh.prolong(h.L, e2g(c, 3)), (4, 2, 2), P)
    for face in [(..., 0), (..., P), (..., 0, slice(1, P)), (..., P, slice(1, P), slice(1, P))]:
        assert np.abs(got[face] - ref[face]).max() <= 1e-13 * np.abs(ref[face]).max()
