"""The one-step FP32 refinement kernel (register tiles) at the edges of its layout:
antennas of a system at and beside 16 and 128 (one to eight warps), odd counts, an
empty cluster, users at and beside 8, 16 and 32, symbols at and beside 4 and 16,
and both residual choices (the FP64 one marks the ill-conditioned systems, which
the generic kernel takes).  Bound of test_gpu_refine after one step:
max(1e-5, 2 kappa 2^-22, 4 (kappa u)^2)."""
import numpy as np
import pytest

import parity
from oracle import llr as ollr
from oracle import lmmse
from paper_1808_04473_gb300 import synth
from test_gpu_refine import ff  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
UNIT = {0: 2.0 ** -24, 2: 2.0 ** -16}

CASES = [  # B, U, C, n_sc, n_sym, cluster sizes, arch (0: PD), precision
    (16, 3, 1, 5, 1, None, 0, 2), (17, 1, 1, 4, 4, None, 0, 0), (34, 8, 2, 7, 5, None, 1, 0),
    (90, 9, 3, 6, 16, [31, 0, 59], 1, 0), (64, 15, 4, 5, 3, None, 1, 2), (127, 16, 1, 3, 14, None, 0, 0),
    (256, 31, 2, 3, 4, None, 1, 2), (256, 32, 1, 2, 16, None, 0, 2), (250, 17, 1, 3, 5, None, 0, 0),
    (8, 5, 4, 6, 2, None, 1, 0),
]


@pytest.mark.parametrize("B,U,C,n_sc,n_sym,sizes,arch,precision", CASES)
@pytest.mark.parametrize("res64", [0, 1])
def test_one_step_edges(ff, B, U, C, n_sc, n_sym, sizes, arch, precision, res64):  # noqa: F811
    p = synth.make_problem(B, U, 1, n_sc, n_sym, snr_db=12.0, bits=4, seed=B + U)
    part = sizes if sizes else [B // C] * C
    dev = torch.device("cuda:0")
    plan = ff.ffeq_plan_create(B, U, C, n_sc, n_sym, arch=arch, precision=precision, llr_bits=4, refine=1,
                               refine_fp64=res64, cluster_sizes=sizes)
    nb = ff.ffeq_workspace_size(plan)
    ws = torch.empty(nb, dtype=torch.uint8, device=dev)
    z = torch.empty((n_sc, n_sym, U), dtype=torch.complex64, device=dev)
    s2 = torch.empty((n_sc, U), device=dev)
    L = torch.empty((n_sc, n_sym, U, 4), device=dev)
    info = torch.full((n_sc, C if arch else 1), -1, dtype=torch.int32, device=dev)
    ff.ffeq_equalize(plan, torch.from_numpy(p.H).to(dev), torch.from_numpy(p.y).to(dev), p.N0, p.Es, z, s2, L, info, ws,
                     nb)
    N0 = float(np.float32(p.N0))
    o = lmmse.equalize_fd(p.H, p.y, N0, p.Es, C, "unbiased", cluster_sizes=part) if arch else \
        lmmse.equalize_pd(p.H, p.y, N0, p.Es, C, "unbiased")
    off = np.concatenate([[0], np.cumsum(part)]) if arch else np.array([0, B])
    kappa = np.array([max(np.linalg.cond(Hk[:, a:b].conj() @ Hk[:, a:b].T + N0 / p.Es * np.eye(U))
                          for a, b in zip(off[:-1], off[1:])) for Hk in p.H.astype(np.complex128)])
    tol = np.maximum(np.maximum(1e-5, 2.0 * 2.0 ** -22 * kappa), 4.0 * (UNIT[precision] * kappa) ** 2)
    parity.check("z", z.cpu().numpy(), o["z"], tol)
    parity.check("sigma2", s2.cpu().numpy(), o["sigma2"], tol)
    parity.check("llr", L.cpu().numpy(), ollr.maxlog_llr(o["z"], o["sigma2"][:, None, :], 4, p.Es), 4 * tol)
    assert (info == 0).all()
