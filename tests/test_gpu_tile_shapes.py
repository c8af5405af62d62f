"""Every tile shape gives the same state bit for bit on grids without open
faces, whichever of the pull forms its kernel uses (loads before or after the
node descriptors): wraps, walls, solids and ragged edges, every storage."""
import numpy as np
import pytest

from paper_2512_12934_gb300 import lbm
from paper_2512_12934_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp16store", "fp64"])
@pytest.mark.parametrize("nx,ny,periodic,solid", [(5, 5, (1, 1), 0.0), (70, 13, (1, 0), 0.06), (129, 37, (0, 1), 0.05),
                                                  (97, 66, (1, 1), 0.04)])
def test_tile_shapes_agree(nx, ny, periodic, solid, precision):
    w = W.random_box(nx, ny, 17, periodic=periodic, solid_frac=solid, G12=0.9, Gw=(0.2, -0.2))
    ref = None
    for v in range(4):
        s = lbm.Solver(w.cfg, w.solid, w.rho, w.u, precision=precision)
        s.set_tile_variant(v)
        s.step(41)
        f = s.populations()
        s.close()
        assert np.isfinite(f).all()
        if ref is None:
            ref = f
        assert np.array_equal(f, ref), v
