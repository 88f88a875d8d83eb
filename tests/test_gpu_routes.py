"""Parity of the kernels that the default dispatch reaches only at some sizes.

* The solve tiles where a CTA of 128 threads takes a subcarrier's systems in several
  passes (more lanes than 128 and more subcarriers than SMs), idle groups in the last
  pass included, and the 512-thread form at the same sizes; with refinement (which
  reads the estimates and inverses they store) and without.  BF16x3, whose FD problems
  always take them.
* The FP32, TF32x3 and FP16x3 contractions and solves of FD problems that the default
  equalizes in one kernel: the 16-warp shape set by the caller, on clusters of their own
  sizes (odd offsets, an empty one), few users and rank-deficient systems.
* The TF32x3 contraction in the 4- and 8-warp shapes that the default takes with many
  subcarriers.

Bounds of test_gpu_parity (with refinement: test_gpu_refine_tile)."""
import numpy as np
import pytest

import parity
from oracle import llr as ollr
from oracle import lmmse
from paper_1808_04473_gb300 import synth
from test_gpu_parity import PREC_TOL, UNIT, _kappa, ff  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(ff, p, C, arch, precision, sizes=None, tuning=None, refine=0):  # noqa: F811
    dev = torch.device("cuda:0")
    plan = ff.ffeq_plan_create(p.B, p.U, C, p.n_sc, p.n_sym, arch=arch, precision=precision, llr_bits=4, refine=refine,
                               cluster_sizes=sizes)
    if tuning:
        ff.ffeq_plan_set_tuning(plan, tuning)
    nb = ff.ffeq_workspace_size(plan)
    ws = torch.empty(nb, dtype=torch.uint8, device=dev)
    z = torch.full((p.n_sc, p.n_sym, p.U), complex("nan"), dtype=torch.complex64, device=dev)
    s2, L = torch.empty((p.n_sc, p.U), device=dev), torch.empty((p.n_sc, p.n_sym, p.U, 4), device=dev)
    info = torch.full((p.n_sc, C if arch else 1), -1, dtype=torch.int32, device=dev)
    ff.ffeq_equalize(plan, torch.from_numpy(p.H).to(dev), torch.from_numpy(p.y).to(dev), p.N0, p.Es, z, s2, L, info, ws,
                     nb)
    assert (info == 0).all()
    return z.cpu().numpy(), s2.cpu().numpy(), L.cpu().numpy()


def _compare(p, got, C, arch, sizes, precision, idx, refined=False):
    f = lmmse.equalize_fd if arch else lmmse.equalize_pd
    kw = dict(cluster_sizes=sizes) if sizes else {}
    o = f(p.H[idx], p.y[idx], float(np.float32(p.N0)), p.Es, C, "unbiased", **kw)
    q = synth.Problem(**{**p.__dict__, "C": C})
    kappa = _kappa(q, arch, idx, sizes)
    tol = np.maximum(PREC_TOL[precision], 2.0 * UNIT[precision] * kappa)
    if refined:   # one step from the BF16x3 systems: test_gpu_refine_tile
        tol = np.maximum(tol, 4.0 * (UNIT[2] * kappa) ** 2)
    parity.check("z", got[0][idx], o["z"], tol)
    parity.check("sigma2", got[1][idx], o["sigma2"], tol)
    parity.check("llr", got[2][idx], ollr.maxlog_llr(o["z"], o["sigma2"][:, None, :], 4, p.Es), 4 * tol)


@pytest.mark.parametrize("B,U,C,n_sc,n_sym", [
    (200, 7, 20, 160, 3), (160, 5, 40, 153, 9), (150, 12, 10, 170, 7), (240, 15, 16, 200, 16), (160, 20, 5, 200, 6),
    (192, 24, 6, 155, 14), (155, 31, 5, 153, 4), (256, 27, 16, 153, 5)])
@pytest.mark.parametrize("refine", [0, 1])
@pytest.mark.parametrize("few", [False, True], ids=["passes", "at-once"])
def test_tiles_in_several_passes(ff, B, U, C, n_sc, n_sym, refine, few):  # noqa: F811
    p = synth.make_problem(B, U, 1, 4 if few else n_sc, n_sym, snr_db=10.0, bits=4, seed=B + U)
    got = _run(ff, p, C, 1, 2, refine=refine)
    idx = np.unique(np.linspace(0, p.n_sc - 1, 24).astype(int))
    _compare(p, got, C, 1, [B // C] * C, 0 if refine else 2, idx, bool(refine))


@pytest.mark.parametrize("precision", [0, 1, 3], ids=["fp32", "tf32x3", "fp16x3"])
@pytest.mark.parametrize("B,U,C,n_sc,n_sym,sizes", [
    (32, 4, 2, 64, 1, None), (33, 5, 3, 9, 2, None), (45, 8, 4, 6, 5, [11, 0, 31, 3]), (51, 7, 3, 4, 9, [17, 0, 34]),
    (40, 20, 5, 7, 4, None), (96, 12, 12, 6, 5, None), (30, 16, 2, 5, 14, [29, 1]), (64, 32, 8, 3, 3, None),
    (128, 9, 32, 20, 8, None)])
def test_contraction_and_solve_of_one_kernel_problems(ff, B, U, C, n_sc, n_sym, sizes, precision):  # noqa: F811
    p = synth.make_problem(B, U, 1, n_sc, n_sym, snr_db=10.0, bits=4, seed=B + 3 * U)
    got = _run(ff, p, C, 1, precision, sizes, tuning=(1, 0))
    _compare(p, got, C, 1, sizes if sizes else [B // C] * C, precision, np.arange(n_sc))


@pytest.mark.parametrize("arch,B,U,C,n_sc,n_sym", [
    (0, 96, 6, 4, 305, 4), (0, 256, 16, 8, 608, 14), (0, 250, 32, 5, 608, 3), (1, 240, 20, 3, 304, 6),
    (1, 192, 18, 6, 320, 9)])
def test_tf32x3_small_cta_shapes(ff, arch, B, U, C, n_sc, n_sym):  # noqa: F811
    p = synth.make_problem(B, U, 1, n_sc, n_sym, snr_db=12.0, bits=4, seed=B + U)
    idx = np.unique(np.linspace(0, n_sc - 1, 24).astype(int))
    for tuning in ((0, 0), (2, 1), (4, 1)):
        try:
            got = _run(ff, p, C, arch, 1, tuning=tuning)
        except ff.FfeqError as e:
            assert e.status == 2 and tuning[0] != 0   # the shape does not fit
            continue
        _compare(p, got, C, arch, [B // C] * C if arch else None, 1, idx)
