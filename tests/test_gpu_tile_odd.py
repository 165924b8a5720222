"""FP64 sweeps over tiles on larger odd grids, whole RHS against the oracle.

These grids have more tiles than the device holds at once, so the tile shape comes
from counting work: 4 or 8 pencils, up to 74 cells along them, runs of 3 to 8
cells, several tiles per pencil with the last one cut short, shorter runs at a
tile's end, and 1 to 5 lanes of the last tile without a pencil.  Bit for bit on
uniform grids; on a refined one, whose tables the library and the oracle compute
independently, within 1e-12 of the fluxes' scale.
"""
import numpy as np
import pytest

import oracle as O
from paper_2409_10729_gb300 import inputs as I
from test_gpu_parity import _stretch, rhs_err

pytestmark = pytest.mark.gpu

CASES = [(2, (131, 97, 75), 5), (2, (131, 97, 75), 3), (2, (173, 131, 95), 5), (2, (1021, 515), 5),
         (3, (97, 83, 61), 5), (3, (701, 402), 5), (4, (61, 59, 83), 5)]


def _problem(nf, n, order, bc):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if nf == 2:
        p, w = I.random_periodic(len(n), list(n), seed=sum(n))
    else:
        p, w = I.random_periodic_n(len(n), list(n), nf, seed=sum(n))
    p = dict(p, weno_order=order, bc=[[bc] * 2 for _ in range(3)])
    return p, w, O.prim_to_cons(p, w)


def _rhs(p, w):
    from paper_2409_10729_gb300 import mfc
    s = mfc.Solver(p, "fp64")
    s.set_state_prim(w)
    L = s.rhs()
    s.close()
    return L


@pytest.mark.parametrize("nf,n,order", CASES, ids=str)
def test_odd_grids_are_the_oracles(nf, n, order):
    p, w, q = _problem(nf, n, order, I.PERIODIC if sum(n) % 2 else I.TRANSMISSIVE)
    assert np.array_equal(_rhs(p, w), O.rhs(p, q))


def test_odd_refined_grid():
    p, w, q = _problem(2, (131, 97, 75), 5, I.TRANSMISSIVE)
    p = _stretch(p, (0, 1, 2))
    assert rhs_err(p, _rhs(p, w), O.rhs(p, q), q, O.max_wavespeed(p, q)).max() <= 1e-12
