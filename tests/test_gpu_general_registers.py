"""General tiles of 32x4 nodes have two register caps, chosen by the lengths of
a step's two lists; the instructions are the same, so a member of a batch on
one side of the line equals the lone device on the other bit for bit."""
import numpy as np
import pytest

from paper_2512_12934_gb300 import lbm
from paper_2512_12934_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("members,large", [(2, True), (9, False)])
def test_batch_members_equal_lone_devices(members, large):
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ws = [W.tjunction(Wc=24 + 2 * i, G12=1.4, Gw=(0.3, -0.3), u_c=0.008) for i in range(members)]
    alone = []
    for w in ws:
        s = lbm.Solver(w.cfg, w.solid, w.rho, w.u)
        st = s.tile_stats()
        assert st["variant"] == 1 and 9 * st["general_tiles"] + 2 * st["fast_tiles"] <= 16 * sms
        s.step(75)
        alone.append(s.populations())
    ms = [lbm.Solver(w.cfg, w.solid, w.rho, w.u) for w in ws]
    b = lbm.Batch(ms)
    i = b.info()
    fits = 2 * i["general_tiles"] <= sms and 9 * i["general_tiles"] + 2 * i["fast_tiles"] <= 16 * sms
    assert fits == large and i["general_tiles"] <= 2 * sms
    b.step(75)
    b.sync()
    for s, f in zip(ms, alone):
        assert np.array_equal(s.populations(), f)
