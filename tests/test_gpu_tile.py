"""FP64 sweeps over tiles: grids whose extents sit on the edges of a tile.

A tile is up to 64 cells of 1, 2 or 4 pencils; the sizes below give single
cells, one cell more or less than a tile, tiles cut short, and pencil counts
that leave lanes of the last tile without a pencil.  RHS and two CFL steps
equal the oracle's bit for bit (the same IEEE operations in the same order).
"""
import numpy as np
import pytest

import oracle as O
from paper_2409_10729_gb300 import inputs as I

pytestmark = pytest.mark.gpu

GRIDS = [(1,), (7,), (8,), (9,), (64,), (65,), (511,), (1, 65), (65, 1), (2, 64), (63, 3), (130, 5), (257, 17),
         (66, 3, 2), (2, 3, 67), (5, 63, 3), (16, 17, 33), (128, 64, 3), (3, 96, 80), (90, 2, 85), (4000, 5)]


@pytest.mark.parametrize("form", ["fp64", "fp64_fast"])
@pytest.mark.parametrize("n", GRIDS, ids=str)
def test_tile_edges(n, form):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_10729_gb300 import mfc
    p, w = I.random_periodic(len(n), list(n), seed=sum(n))
    if sum(n) % 2:
        p = dict(p, bc=[[I.TRANSMISSIVE] * 2 for _ in range(3)])
    q = O.prim_to_cons(p, w)
    s = mfc.Solver(p, form)
    s.set_state_prim(w)
    assert np.array_equal(s.rhs(), O.rhs(p, q))
    t = s.step_rk3(0.4, 2)
    qo, to = O.run_cfl(p, q, 0.4, 2)
    assert np.array_equal(s.get_state(), qo) and t == to
    s.close()


@pytest.mark.parametrize("order", [5, 3])
@pytest.mark.parametrize("scale", [1e-90, 1e-60, 1e45, 1e70])
def test_far_units(scale, order):
    """Densities and pressures far from 1: the smoothness indicators, their squares
    and the weights leave the range of the integer products and quotients, and
    the FP64 instructions answer -- still the oracle's bits."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_10729_gb300 import mfc
    p, w = I.random_periodic(2, [40, 24], seed=5)
    w = w.copy()
    w[:2] *= scale
    w[4] *= scale
    p = dict(p, weno_order=order, pi_inf=[x * scale for x in p["pi_inf"]])
    q = O.prim_to_cons(p, w)
    s = mfc.Solver(p, "fp64")
    s.set_state_prim(w)
    assert np.array_equal(s.get_state(), q)
    assert np.array_equal(s.rhs(), O.rhs(p, q))
    t = s.step_rk3(0.4, 2)
    qo, to = O.run_cfl(p, q, 0.4, 2)
    assert np.array_equal(s.get_state(), qo) and t == to
    s.close()
