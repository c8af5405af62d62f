"""Reading the macroscopic fields: the device-destination kernels, the staged
host reads and the copy route for unaligned destinations give the same values
(2D and 3D, all precisions, ragged extents, solids)."""
import numpy as np
import pytest

from paper_2512_12934_gb300 import lbm
from paper_2512_12934_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _cases():
    return [W.channel(nx=65, ny=17, R=4, xc=20, G12=1.2), W.random_box(5, 5, 3),
            W.random_box(257, 9, 4, solid_frac=0.2), W.duct3(nx=33, ny=9, nz=7, R=2.0, G12=1.2),
            W.random_box3(65, 5, 6, 5, solid_frac=0.2)]


@pytest.mark.parametrize("precision", ["fp32", "fp16store", "fp64"])
@pytest.mark.parametrize("case", range(5))
def test_device_host_and_unaligned_reads_agree(case, precision):
    import torch

    w = _cases()[case]
    s = lbm.Solver(w.cfg, w.solid, w.rho, w.u, precision=precision)
    try:
        s.step(3)
        r64, u64 = s.macros()
        r32, u32 = s.macros_f32()
        assert np.array_equal(r32, r64.astype(np.float32)) and np.array_equal(u32, u64.astype(np.float32))
        if w.solid is not None:
            assert not r64[:, w.solid != 0].any() and not u64[:, w.solid != 0].any()
        nr, nu = r32.size, u32.size
        for shift in (0, 2):  # bytes off the allocation's start: 2 is not a float boundary
            raw = torch.full((4 * (nr + nu) + 64,), 0x7F, dtype=torch.uint8, device="cuda")
            base = raw.data_ptr() + shift
            s.macros_f32(base, base + 4 * nr, device=True)
            got = raw.cpu().numpy()
            assert np.array_equal(got[shift:shift + 4 * nr].view(np.float32), r32.reshape(-1))
            assert np.array_equal(got[shift + 4 * nr:shift + 4 * (nr + nu)].view(np.float32), u32.reshape(-1))
            assert (got[shift + 4 * (nr + nu):] == 0x7F).all() and (got[:shift] == 0x7F).all()
    finally:
        s.close()


@pytest.mark.parametrize("three", [False, True])
def test_a_diverged_run_reports_and_leaves_the_destination(three):
    import torch

    w = W.random_box3(33, 6, 5, 7) if three else W.random_box(40, 12, 7)
    s = lbm.Solver(w.cfg, w.solid, w.rho, w.u)
    try:
        f = s.populations()
        f[0, 0].flat[3] = np.nan
        s.set_populations(f)
        s.step(2)
        rho = torch.full((2, *s.shape), 5.0, device="cuda")
        u = torch.full((s.dim, *s.shape), 5.0, device="cuda")
        with pytest.raises(lbm.LbmError) as e:
            s.macros_f32(rho.data_ptr(), u.data_ptr(), device=True)
        assert e.value.status == 4
        assert bool((rho == 5).all()) and bool((u == 5).all())
    finally:
        s.close()
