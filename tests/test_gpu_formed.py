"""The FP32 kernels that form the local systems in registers from staged inputs
(training forward, its adjoint, the adjoint through the optimal weights, the fused
FD equalization) where their layouts change: users at and beside the padded sizes
8, 16 and 32, right-hand sides at and beside 4, 8 and 16, odd and empty clusters
(8-byte copies, antennas one at a time), more clusters than lane groups (several
passes), a single subcarrier.  Bounds of test_gpu_adjoint and test_gpu_parity."""
import numpy as np
import pytest

import parity
from oracle import adjoint, lmmse
from oracle import llr as ollr
from paper_1808_04473_gb300 import synth
from test_gpu_adjoint import _optimal, _relmax, _run, ff  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [  # B, U, C, n_sc, n_sym, cluster sizes
    (2, 1, 2, 1, 1, None), (33, 5, 3, 9, 4, None), (45, 8, 5, 6, 5, None), (64, 9, 32, 3, 8, None),
    (51, 7, 3, 4, 9, [17, 0, 34]), (96, 16, 6, 5, 16, None), (95, 17, 5, 3, 1, None), (63, 15, 3, 1, 6, [20, 21, 22]),
    (128, 31, 16, 3, 5, None), (128, 32, 4, 2, 16, None), (128, 4, 32, 7, 3, None),
]
IDS = [f"{c[0]}-{c[1]}-{c[2]}-{c[3]}-{c[4]}{'' if c[5] is None else '-sizes'}" for c in CASES]


@pytest.mark.parametrize("B,U,C,n_sc,n_sym,sizes", CASES, ids=IDS)
def test_training_edges(ff, B, U, C, n_sc, n_sym, sizes):  # noqa: F811
    p = synth.make_problem(B, U, 1, n_sc, n_sym, snr_db=10.0, bits=2, seed=B + C)
    rng = np.random.default_rng(B + C)
    rho = ((p.N0 / p.Es) * rng.uniform(0.5, 2.0, C)).astype(np.float32)
    nu = (rng.uniform(0.5, 1.5, (C, U)) / C).astype(np.float32)
    kw = dict(cluster_sizes=sizes) if sizes else dict(cluster_sizes=[B // C] * C)
    z0, _ = adjoint.fd_train_forward(p.H, p.y, rho.astype(np.float64), nu.astype(np.float64), **kw)
    gz = 2.0 * (z0 - p.s) / z0.size
    g = _run(ff, p, rho, nu, C, gz, sizes)
    parity.check("z", g["z"], z0, 1e-5)
    gH, gy, grho, gnu = adjoint.fd_train_backward(p.H, p.y, rho.astype(np.float64), nu.astype(np.float64),
                                                  gz.astype(np.complex64).astype(np.complex128), **kw)
    parity.check("gH", g["gH"], gH, 1e-3)
    parity.check("gy", g["gy"], gy, 1e-3)
    for name, ref in (("grho", grho), ("gnu", gnu)):
        assert _relmax(g[name], ref) <= 1e-3, (name, _relmax(g[name], ref))


@pytest.mark.parametrize("B,U,C,n_sc,n_sym,sizes", CASES, ids=IDS)
def test_optimal_adjoint_edges(ff, B, U, C, n_sc, n_sym, sizes):  # noqa: F811
    p = synth.make_problem(B, U, 1, n_sc, n_sym, snr_db=8.0, bits=2, seed=B + 3 * U)
    N0 = float(np.float32(p.N0))
    kw = dict(cluster_sizes=sizes if sizes else [B // C] * C)
    z0 = lmmse.equalize_fd(p.H, p.y, N0, p.Es, C, "unbiased", **kw)["z"]
    gz = 2.0 * (z0 - p.s) / z0.size
    gH, gy = _optimal(ff, p, C, gz, sizes)
    oH, oy = adjoint.fd_optimal_backward(p.H, p.y, N0, p.Es, C, gz.astype(np.complex64).astype(np.complex128), **kw)
    parity.check("gH", gH, oH, 1e-3)
    parity.check("gy", gy, oy, 1e-3)


@pytest.mark.parametrize("B,U,C,n_sc,n_sym,sizes", CASES, ids=IDS)
@pytest.mark.parametrize("estimate", [0, 1], ids=["unbiased", "literal"])
def test_fused_equalization_edges(ff, B, U, C, n_sc, n_sym, sizes, estimate):  # noqa: F811
    p = synth.make_problem(B, U, 1, n_sc, n_sym, snr_db=10.0, bits=4, seed=B + 5 * U)
    dev = torch.device("cuda:0")
    plan = ff.ffeq_plan_create(B, U, C, n_sc, n_sym, arch=ff.FD, llr_bits=4, estimate=estimate, cluster_sizes=sizes)
    nb = ff.ffeq_workspace_size(plan)
    ws = torch.empty(nb, dtype=torch.uint8, device=dev)
    z = torch.empty((n_sc, n_sym, U), dtype=torch.complex64, device=dev)
    s2 = torch.empty((n_sc, U), device=dev)
    L = torch.empty((n_sc, n_sym, U, 4), device=dev)
    info = torch.full((n_sc, C), -1, dtype=torch.int32, device=dev)
    ff.ffeq_equalize(plan, torch.from_numpy(p.H).to(dev), torch.from_numpy(p.y).to(dev), p.N0, p.Es, z, s2, L, info, ws,
                     nb)
    o = lmmse.equalize_fd(p.H, p.y, float(np.float32(p.N0)), p.Es, C, "unbiased" if estimate == 0 else "literal",
                          cluster_sizes=sizes if sizes else [B // C] * C)
    # FP32 unit roundoff times the largest condition number of the systems solved (test_gpu_parity).
    rho, off = p.N0 / p.Es, np.concatenate([[0], np.cumsum(sizes if sizes else [B // C] * C)])
    kappa = [max(np.linalg.cond(Hk[:, a:b].conj() @ Hk[:, a:b].T + rho * np.eye(U)) for a, b in zip(off[:-1], off[1:]))
             for Hk in p.H.astype(np.complex128)]
    tol = np.maximum(1e-5, 2.0 * 2.0 ** -22 * np.array(kappa))
    parity.check("z", z.cpu().numpy(), o["z"], tol)
    parity.check("sigma2", s2.cpu().numpy(), o["sigma2"], tol)
    parity.check("llr", L.cpu().numpy(), ollr.maxlog_llr(o["z"], o["sigma2"][:, None, :], 4, p.Es), 4 * tol)
    assert (info == 0).all()
