"""D3Q19 grids with interior collide tiles, whose density boxes come as one
tensor copy (nx >= 66, ny >= 10, nz >= 6), beside ragged edge tiles, whose boxes
are staged by loads: both storages against the FP64 oracle, graph replay against
plain launches, and the two kinds of tile against one another (a periodic box
rolled so that every node changes its kind of tile gives the same state, bit
for bit)."""
import numpy as np
import pytest

from oracle import oracle3d as O3
from paper_2512_12934_gb300 import workloads as W
from test_gpu_d3q19 import TOL32, check, lbm, rel, run_both  # noqa: F401
from test_gpu_d3q19_graphs import run

pytestmark = pytest.mark.gpu


def case(name):
    if name == "duct":
        return W.duct3(nx=100, ny=14, nz=11, R=3.0, xc=24.0, u_max=0.02, G12=1.2, Gw=(0.2, -0.2)), 0.02
    if name == "solids":
        return W.random_box3(70, 13, 9, seed=12, periodic=(1, 0, 1), solid_frac=0.06, G12=1.0, Gw=(0.3, -0.3),
                             nu=(0.12, 0.2), u_amp=0.01, rho_lo=0.4, rho_hi=1.0), 0.01
    return W.random_box3(70, 11, 7, seed=11, G12=0.6, nu=(0.1, 0.2), u_amp=0.05, rho_lo=0.6, rho_hi=1.0), 0.05


@pytest.mark.parametrize("name", ["duct", "solids", "box"])
def test_fp32_matches_the_oracle(lbm, name):  # noqa: F811
    w, us = case(name)
    g, r = run_both(lbm, w, 100)
    check(g, r, TOL32, name, u_scale=us)


@pytest.mark.parametrize("name", ["duct", "solids"])
def test_fp16_storage_error_is_bounded(lbm, name):  # noqa: F811
    """The bounds of the smaller grids' FP16 test; that on the minor phase for the
    device, whose phases are apart (in the mixed box a component is depleted
    beside major-phase nodes)."""
    w, us = case(name)
    (rg, ug, d, _), (ro, uo, sc, _) = run_both(lbm, w, 100, precision="fp16store")
    assert rel(rg[0] + rg[1], ro[0] + ro[1]) < 2e-4
    if name == "duct":
        minor = (ro > 0) & (ro < 0.01)
        assert minor.any() and np.abs(rg - ro)[minor].max() < 1e-5
    assert np.abs(ug - uo).max() < 5e-3 * max(np.abs(uo).max(), us)
    assert np.allclose(d["mass"], sc["mass"], rtol=2e-4)


@pytest.mark.parametrize("precision", ["fp32", "fp16store"])
def test_graph_replay_equals_plain_launches(precision):
    w, _ = case("duct")
    f0, (r0, u0), d0 = run(w, precision, False, (55,))
    for runs in ((55,), (1, 17, 37)):
        f1, (r1, u1), d1 = run(w, precision, True, runs)
        assert np.array_equal(f0, f1) and np.array_equal(r0, r1) and np.array_equal(u0, u1)
        assert d0 == d1


@pytest.mark.parametrize("precision", ["fp32", "fp16store"])
def test_copied_and_staged_boxes_agree(lbm, precision):  # noqa: F811
    w = W.random_box3(100, 14, 11, seed=21, solid_frac=0.04, G12=0.9, Gw=(0.2, -0.2), nu=(0.12, 0.2), u_amp=0.01,
                      rho_lo=0.4, rho_hi=1.0)
    solid = np.asarray(w.solid).reshape(11, 14, 100)
    out = []
    for shift in ((0, 0, 0), (5, 7, 50), (6, 3, 29)):
        roll = lambda a, s=shift: np.ascontiguousarray(np.roll(a, s, axis=(-3, -2, -1)))  # noqa: E731
        back = tuple(-s for s in shift)
        s = lbm.Solver(w.cfg, roll(solid), roll(w.rho), roll(w.u), precision=precision)
        s.step(23)
        f, (rho, u) = s.populations(), s.macros()
        s.close()
        out.append([np.roll(a, back, axis=(-3, -2, -1)) for a in (f, rho, u)])
    assert np.isfinite(out[0][0]).all()
    for o in out[1:]:
        for a, b in zip(o, out[0]):
            assert np.array_equal(a, b)
