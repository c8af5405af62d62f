"""Steps recorded into a caller's stream capture: runs of every length a step
graph would serve are recorded as plain launches, and a replay of the caller's
graph leaves the state that the same steps leave when run at once, bit for
bit (2D, batch and 3D; before and after the context has graphs of its own).
Steps on one stream while another is being captured run at once, graphs of their
own included, and leave that capture alone."""
import numpy as np
import pytest

from paper_2512_12934_gb300 import lbm
from paper_2512_12934_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def make(kind, stream):
    if kind == "3d":
        w = W.laplace3(n=20, R=5.0, G12=1.2)
        s = lbm.Solver(w.cfg, w.solid, w.rho, w.u, stream=stream)
        return s, [s]
    ws = [W.channel(nx=130, ny=30, R=6, xc=40, u_max=0.02, G12=1.4, Gw=(0.3, -0.3)),
          W.laplace(nx=70, ny=50, R=12, G12=1.2)]
    if kind == "2d":
        ws = ws[:1]
    ms = [lbm.Solver(w.cfg, w.solid, w.rho, w.u, stream=stream) for w in ws]
    return (lbm.Batch(ms, stream=stream) if kind == "batch" else ms[0]), ms


@pytest.mark.parametrize("warm", [0, 76])
@pytest.mark.parametrize("n", [3, 10, 40])
@pytest.mark.parametrize("kind", ["2d", "batch", "3d"])
def test_captured_steps_replay(kind, n, warm):
    import torch

    plain, pm = make(kind, None)
    plain.step(warm)
    plain.step(n)
    plain.sync()
    st = torch.cuda.Stream()
    run, rm = make(kind, st.cuda_stream)
    run.step(warm)
    run.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        run.step(n)
    g.replay()
    torch.cuda.synchronize()
    run.sync()
    for a, b in zip(pm, rm):
        assert np.array_equal(a.populations(), b.populations())
    run.step(n)  # and the context steps on by itself
    plain.step(n)
    run.sync()
    plain.sync()
    for a, b in zip(pm, rm):
        assert np.array_equal(a.populations(), b.populations())


@pytest.mark.parametrize("mode", ["global", "thread_local", "relaxed"])
@pytest.mark.parametrize("kind", ["2d", "batch", "3d"])
def test_steps_beside_a_capture(kind, mode):
    import torch

    runs = (10, 10, 10, 40)
    plain, pm = make(kind, None)
    for n in runs:
        plain.step(n)
    plain.sync()
    captured, own = torch.cuda.Stream(), torch.cuda.Stream()
    run, rm = make(kind, own.cuda_stream)
    run.sync()
    x = torch.zeros(100, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=captured, capture_error_mode=mode):
        x += 1
        for n in runs:
            run.step(n)
        x += 1
    run.sync()
    for a, b in zip(pm, rm):
        assert np.array_equal(a.populations(), b.populations())
    g.replay()
    torch.cuda.synchronize()
    assert float(x[0]) == 2.0
