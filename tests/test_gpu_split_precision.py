"""GPU: the digit-split FP64 kernels keep FP64 precision where values of very different size meet.

Every bound is relative to what a value is formed from, not to the largest value around it.
"""
import numpy as np
import pytest

import synthetic as syn
from oracle import dg, schwarz
from tests.helpers import e2g, elem_shape, from_dev, to_dev

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
