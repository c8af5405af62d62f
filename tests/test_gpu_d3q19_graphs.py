"""D3Q19 step runs replayed from two-branch graphs are the plain launches, bit
for bit: with and without open faces, every storage, runs that start on either
ping-pong parity, and a reset between them."""
import numpy as np
import pytest

from paper_2512_12934_gb300 import lbm
from paper_2512_12934_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def run(w, precision, graphs, runs):
    s = lbm.Solver(w.cfg, w.solid, w.rho, w.u, precision=precision)
    try:
        s.set_graph_mode(graphs)
        s.step(18)
        s.reset(w.rho, w.u)
        for n in runs:
            s.step(n)
        d = s.diagnostics()
        return s.populations(), s.macros(), (d["lambda"], d["chi"], d["Qin"], d["Qout"], d["step"], d["launches"])
    finally:
        s.close()


@pytest.mark.parametrize("precision", ["fp32", "fp16store", "fp64"])
@pytest.mark.parametrize("name", ["duct", "droplet"])
def test_graph_replay_equals_plain_launches(name, precision):
    w = (W.duct3(nx=40, ny=9, nz=8, R=2.5, xc=10.0, u_max=0.02, G12=1.2) if name == "duct"
         else W.laplace3(n=20, R=5.0, G12=1.2))
    f0, (r0, u0), d0 = run(w, precision, False, (55,))
    for runs in ((55,), (1, 17, 37)):
        f1, (r1, u1), d1 = run(w, precision, True, runs)
        assert np.array_equal(f0, f1) and np.array_equal(r0, r1) and np.array_equal(u0, u1)
        assert d0 == d1
