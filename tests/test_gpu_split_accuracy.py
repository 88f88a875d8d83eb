"""Accuracy of the TF32x3 contraction in its small-CTA shapes: the default and shapes
2 and 4 split a cluster's antennas among fewer warps than shape 1, so each warp adds
more k-steps.  The RMS error of the local Gram matrices and matched filters against
64 bits must not exceed shape 1's by more than a tenth (sums rounded to nearest grow
with the square root of their terms only, and shape 1 adds as many partial sums; the
spread of the ratio over the entries here is below a hundredth).  Sizes: enough
subcarriers for the default to leave shape 1, antennas that fill no k-step, K-parts
of one and of many k-steps, and clusters of their own."""
import numpy as np
import pytest

from paper_1808_04473_gb300 import synth
from test_gpu_parity import ff  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [  # arch (0: PD), B, U, C, n_sc, n_sym
    (0, 96, 6, 4, 608, 4), (0, 100, 12, 5, 333, 7), (0, 256, 8, 1, 320, 4), (0, 256, 16, 8, 608, 14),
    (0, 250, 20, 5, 608, 10), (0, 256, 32, 4, 608, 3), (1, 240, 20, 3, 304, 6), (1, 256, 24, 2, 304, 9),
    (1, 90, 32, 1, 304, 1),
]


def _error(D, H, y, arch, C):
    """RMS of D - D64 over RMS of D64, D64[v][u] = sum_b conj(H[u][b]) W[v][b], W = [H; y]."""
    n_sc, U, B = H.shape
    parts = C if arch else 1
    h = H.to(torch.complex128).reshape(n_sc, U, parts, B // parts)
    w = torch.cat([H, y], 1).to(torch.complex128).reshape(n_sc, -1, parts, B // parts)
    ref = torch.einsum("kvcb,kucb->kcvu", w, h.conj())
    return float(((D - ref).abs().square().sum() / ref.abs().square().sum()).sqrt())


@pytest.mark.parametrize("arch,B,U,C,n_sc,n_sym", CASES)
def test_small_cta_shapes_are_as_accurate_as_shape_1(ff, arch, B, U, C, n_sc, n_sym):  # noqa: F811
    p = synth.make_problem(B, U, C, n_sc, n_sym, snr_db=12.0, bits=4, seed=B + U + n_sym)
    dev = torch.device("cuda:0")
    H, y = torch.from_numpy(p.H).to(dev), torch.from_numpy(p.y).to(dev)
    plan = ff.ffeq_plan_create(B, U, C, n_sc, n_sym, arch=arch, precision=ff.TF32X3)
    nb = ff.ffeq_workspace_size(plan)
    err = {}
    for shape in ((1, 0), (0, 0), (2, 0), (2, 1), (4, 0), (4, 1)):
        try:
            ff.ffeq_plan_set_tuning(plan, shape)
        except ff.FfeqError as e:
            assert e.status == 2 and shape[0] in (2, 4)   # does not fit
            continue
        ws = torch.full((nb // 8,), complex("nan"), dtype=torch.complex64, device=dev)
        ff.ffeq_local_preprocess(plan, H, y, ws, nb)
        err[shape] = _error(ws.view(n_sc, C if arch else 1, U + n_sym, U), H, y, arch, C)
    assert (2, 1) in err or (4, 1) in err
    for shape, e in err.items():
        assert e <= 1.1 * err[(1, 0)], (shape, e, err[(1, 0)])


@pytest.mark.parametrize("arch", [0, 1], ids=["PD", "FD"])
def test_batch_is_as_accurate_as_shape_1(ff, arch):  # noqa: F811
    """A batch of enough units for its 8-warp shape, one size: sigma^2 against a uniform plan's on shape 1."""
    B, U, C, n_sc, n_sym = 256, 16, 2, 500, 14
    p = synth.make_problem(B, U, C, n_sc, n_sym, snr_db=12.0, bits=4, seed=4)
    dev = torch.device("cuda:0")
    H, y = torch.from_numpy(p.H).to(dev), torch.from_numpy(p.y).to(dev)
    h = H.to(torch.complex128).reshape(n_sc, U, C if arch else 1, -1).transpose(1, 2)
    A = torch.linalg.inv(h.conj() @ h.mT + p.N0 / p.Es * torch.eye(U, device=dev))
    a = torch.diagonal(A, dim1=-2, dim2=-1).real
    ref = 1.0 / ((1.0 - p.N0 / p.Es * a) / (p.N0 * a)).sum(1)
    err = lambda s: float(((s.double() - ref).square().sum() / ref.square().sum()).sqrt())  # noqa: E731
    z, s2 = torch.empty((n_sc, n_sym, U), dtype=torch.complex64, device=dev), torch.empty((n_sc, U), device=dev)
    plan = ff.ffeq_plan_create(B, U, C, n_sc, n_sym, arch=arch, precision=ff.TF32X3)
    ff.ffeq_plan_set_tuning(plan, (1, 0))
    nb = ff.ffeq_workspace_size(plan)
    ws = torch.empty(nb, dtype=torch.uint8, device=dev)
    ff.ffeq_local_preprocess(plan, H, y, ws, nb)
    ff.ffeq_fuse_equalize(plan, ws, nb, p.N0, p.Es, z, s2)
    uniform = err(s2)
    cfg, inst = ff.pack_batch([(B, U, C, n_sc, n_sym, p.N0, p.Es)], arch=arch, precision=ff.TF32X3)
    batch = ff.ffeq_batch_create(cfg, inst)
    nb = ff.ffeq_batch_workspace_size(batch)
    ws = torch.empty(nb, dtype=torch.uint8, device=dev)
    ff.ffeq_batch_upload(batch, ws, nb)
    info = torch.zeros(max(cfg.info_elems, 1), dtype=torch.int32, device=dev)
    ff.ffeq_batch_equalize(batch, H, y, z, s2, None, info if cfg.info_elems else None, ws, nb)
    torch.cuda.synchronize()
    assert err(s2) <= 1.1 * uniform, (err(s2), uniform)
