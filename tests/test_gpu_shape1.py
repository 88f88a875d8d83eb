"""A contraction shape that the caller sets is the one that runs, also where the default
shape is the one-kernel FP32 equalization: the workspace then holds the local systems of
that shape, and ffeq_fuse_equalize of them gives the outputs of ffeq_equalize bit for
bit; the default leaves the workspace as it was.  The autotuner returns a contraction
shape in every case, and what it decided about the one kernel holds until a shape is
set."""
import numpy as np
import pytest

import parity
from oracle import lmmse
from paper_1808_04473_gb300 import synth
from test_gpu_parity import _bound, ff  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1, 3], ids=["fp32", "tf32x3", "fp16x3"])
@pytest.mark.parametrize("B,U,C,n_sc,n_sym", [(32, 4, 2, 64, 1), (48, 7, 3, 5, 3), (128, 12, 8, 330, 8)])
def test_set_shape_runs_its_contraction(ff, B, U, C, n_sc, n_sym, precision):  # noqa: F811
    p = synth.make_problem(B, U, C, n_sc, n_sym, snr_db=10.0, bits=4, seed=B + U)
    dev = torch.device("cuda:0")
    H, y = torch.from_numpy(p.H).to(dev), torch.from_numpy(p.y).to(dev)
    plan = ff.ffeq_plan_create(B, U, C, n_sc, n_sym, arch=ff.FD, precision=precision)
    nb = ff.ffeq_workspace_size(plan)
    z = [torch.empty((n_sc, n_sym, U), dtype=torch.complex64, device=dev) for _ in range(2)]
    s2 = [torch.empty((n_sc, U), device=dev) for _ in range(2)]
    bits = lambda t: t.contiguous().view(torch.uint8)  # noqa: E731
    o = lmmse.equalize_fd(p.H, p.y, float(np.float32(p.N0)), p.Es, C, "unbiased")
    tol = _bound(p, 1, precision)

    def equalize():
        ws = torch.full((nb,), 255, dtype=torch.uint8, device=dev)
        ff.ffeq_equalize(plan, H, y, p.N0, p.Es, z[0], s2[0], None, None, ws, nb)
        parity.check("z", z[0].cpu().numpy(), o["z"], tol)
        parity.check("sigma2", s2[0].cpu().numpy(), o["sigma2"], tol)
        return ws

    assert ff.ffeq_plan_single_launch(plan)
    assert (equalize() == 255).all()
    for shape in ((1, 0), (1, 1), (2, 0), (4, 0), (5, 0)):
        try:
            ff.ffeq_plan_set_tuning(plan, shape)
        except ff.FfeqError as e:
            assert e.status == 2 and shape[0] != 1
            continue
        ws = equalize()
        alone = torch.full((nb,), 255, dtype=torch.uint8, device=dev)
        ff.ffeq_local_preprocess(plan, H, y, alone, nb)
        assert (ws == alone).all() and not (ws == 255).all(), shape
        ff.ffeq_fuse_equalize(plan, ws, nb, p.N0, p.Es, z[1], s2[1])
        assert (bits(z[0]) == bits(z[1])).all() and (bits(s2[0]) == bits(s2[1])).all(), shape
    ws = torch.full((nb,), 255, dtype=torch.uint8, device=dev)
    t = ff.ffeq_plan_autotune(plan, H, y, p.N0, p.Es, z[0], s2[0], None, None, ws, nb, reps=3)
    assert 1 <= t[0] <= 7 and 1 <= t[1] <= 3 and ff.ffeq_plan_get_tuning(plan) == t
    assert (equalize() == 255).all() == ff.ffeq_plan_single_launch(plan)
    ff.ffeq_plan_set_tuning(plan, t)
    assert not ff.ffeq_plan_single_launch(plan) and not (equalize() == 255).all()
