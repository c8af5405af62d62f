"""The tile shape a batch takes when its members' defaults differ: the same
for every order of the members, so that a member's results depend neither on
the order nor on the other members; a shape the caller set wins."""
import itertools

import numpy as np
import pytest

from paper_2512_12934_gb300 import lbm
from paper_2512_12934_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def devices():
    return {"channel": W.channel(nx=130, ny=30, R=6, xc=40, u_max=0.02, G12=1.4, Gw=(0.3, -0.3)),
            "tjunction": W.tjunction(Wc=12, length_factor=12, Wd=6, side_len=10, x_side=30, G12=1.4, Gw=(0.3, -0.3)),
            "laplace": W.laplace(nx=70, ny=50, R=12, G12=1.2)}


def solver(w):
    return lbm.Solver(w.cfg, w.solid, w.rho, w.u)


def test_default_tiles_do_not_depend_on_member_order():
    ws = devices()
    alone = {}
    for name, w in ws.items():
        s = solver(w)
        s.step(200)
        alone[name] = (s.tile_stats()["variant"], s.populations())
    assert alone["tjunction"][0] == 1 and alone["channel"][0] == alone["laplace"][0] == 0
    for order in itertools.permutations(ws):
        ms = {name: solver(ws[name]) for name in order}
        b = lbm.Batch(list(ms.values()))
        assert b.info()["variant"] == 1
        b.step(200)
        b.sync()
        for name, s in ms.items():
            f, f0 = s.populations(), alone[name][1]
            if name == "channel":  # other tiles than alone: chi's FP64 partials are grouped otherwise
                assert np.abs(f - f0).max() <= 1e-5 * np.abs(f0).max(), order
            else:
                assert np.array_equal(f, f0), (order, name)
        b.close()
        # a re-tiled member does not hand its shape to its next batch
        b = lbm.Batch([ms["laplace"], ms["channel"]])
        assert b.info()["variant"] == 0
        b.close()


@pytest.mark.parametrize("first", [True, False])
def test_a_set_tile_shape_wins(first):
    ws = devices()
    a, t = solver(ws["channel"]), solver(ws["tjunction"])
    a.set_tile_variant(2)
    b = lbm.Batch([a, t] if first else [t, a])
    assert b.info()["variant"] == 2
    b.close()
