"""The default tile shape of closed FP64 grids: the shape whose busiest SM has
the fewest tile rows; the state does not depend on it."""
import numpy as np
import pytest

from paper_2512_12934_gb300 import lbm
from paper_2512_12934_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(64, 64), (100, 100), (150, 160), (200, 200), (256, 256), (400, 390)])
def test_closed_fp64_grids_balance_their_tiles(nx, ny):
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    up = lambda a, b: -(-a // b)  # noqa: E731
    rows8 = 2 * up(up(nx, 32) * up(ny, 8), sms)
    rows4 = up(up(nx, 32) * up(ny, 4), sms)
    w = W.laplace(nx=nx, ny=ny, R=min(nx, ny) // 5, G12=1.2)
    out = []
    for v in (None, 0, 1):
        s = lbm.Solver(w.cfg, w.solid, w.rho, w.u, precision="fp64")
        if v is None:
            assert s.tile_stats()["variant"] == (1 if rows4 < rows8 else 0)
        else:
            s.set_tile_variant(v)
        s.step(11)
        out.append(s.populations())
        s.close()
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])


def test_closed_fp64_batches_balance_all_tiles():
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    up = lambda a, b: -(-a // b)  # noqa: E731
    for sizes in ([100] * 2, [100] * 5, [128, 160, 160], [64] * 11):
        ms = []
        for n in sizes:
            w = W.laplace(nx=n, ny=n, R=n // 5, G12=1.2)
            ms.append(lbm.Solver(w.cfg, w.solid, w.rho, w.u, precision="fp64"))
        t8, t4 = (sum(up(n, 32) * up(n, r) for n in sizes) for r in (8, 4))
        b = lbm.Batch(ms)
        assert b.info()["variant"] == (1 if up(t4, sms) < 2 * up(t8, sms) else 0)
        b.close()
