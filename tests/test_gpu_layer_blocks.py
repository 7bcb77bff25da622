"""The exact layer blocks of lines beyond 160 sites (slices of 32), where their inverse runs
in 64 x 64 tiles with 32 x 32 pivots: lines of 161 (33 sites in the last tile, 1 in the
last pivot), 193, 224 (half a tile), 320 (whole tiles) and 1024, the longest.  One
interface line: its block is S itself, so an inverse that is exact to complex64 leaves
two or three COCG iterations to 1e-13 (FP64) and one or two to 1e-5 (a mixed solve);
converged results alone would not show a wrong inverse."""
import numpy as np
import pytest

from paper_1102_3137_gb300 import dyson as D
from paper_1102_3137_gb300 import inputs as I
from parity_util import plan_for, wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx", [161, 193, 224, 320, 1024])
@pytest.mark.parametrize("precision", [D.DYSON_FP64, D.DYSON_MIXED])
def test_long_line_inverse_at_tile_edges(Lx, precision):
    from paper_1102_3137_gb300 import build
    build.build()
    D.load()
    w = wl((Lx, 65), 2, 4, K=3, beta=10.0)
    omega, V, sigma, q1 = I.make_inputs(w)
    pl = plan_for(w, precision, precond=D.DYSON_PRECOND_LAYER)
    st = np.zeros(w.K, np.int32)
    pl.solve(omega, V, sigma, q1, status=st)
    info = pl.info(w.K)
    assert np.all(st == 0)
    if precision == D.DYSON_FP64:
        assert np.all(info["iters"] / info["steps"] <= 3.5)
    else:                                    # a solve per X-matvec and one per refinement pass
        assert np.all(info["iters"] <= 2 * (info["steps"] + info["refines"]))
    pl.close()
