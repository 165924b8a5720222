"""The mixed form's two kernels of a sweep give the same bits.

Small launches take the lean kernel, large ones the full one, so a periodic state
and the same state repeated over a larger grid of the same widths run different
kernels; the right-hand sides are equal cell by cell (WENO3 and the non-uniform
reconstruction carry nothing from cell to cell, so no tolerance is needed).
"""
import numpy as np
import pytest

from paper_2409_10729_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _rhs(p, w):
    from paper_2409_10729_gb300 import mfc
    s = mfc.Solver(p, "mixed")
    s.set_state_prim(w)
    out = s.rhs()
    s.close()
    return out


@pytest.mark.parametrize("n,reps,refined", [((64, 32), (10, 10), False), ((61, 33), (10, 10), False),
                                            ((32, 32, 32), (2, 2, 2), False), ((31, 17, 22), (3, 5, 4), False),
                                            ((640, 32), (1, 10), True), ((96, 32, 16), (1, 3, 6), True)])
def test_small_and_repeated_grids_agree(n, reps, refined):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nd, dx = len(n), 2.0 ** -6   # widths exact on both grids
    p, w = I.random_periodic(nd, list(n), seed=11)
    w = np.ascontiguousarray(w)
    edges = [np.cumsum(np.r_[0.0, dx * (1.0 + 0.25 * np.sin(2 * np.pi * np.arange(n[0]) / n[0]))])] + [None] * (nd - 1)

    def problem(k):
        q = dict(p, n=[n[d] * k[d] for d in range(nd)] + [1] * (3 - nd), lo=[0.0] * 3,
                 hi=[n[d] * k[d] * dx for d in range(nd)] + [1.0] * (3 - nd))
        return dict(q, edges=edges) if refined else dict(q, weno_order=3)

    tile = (1,) + (1,) * (3 - nd) + tuple(reps[::-1])
    small = _rhs(problem((1,) * nd), w)
    large = _rhs(problem(reps), np.ascontiguousarray(np.tile(w, tile)))
    assert np.array_equal(large, np.tile(small, tile))
