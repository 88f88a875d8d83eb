"""The fused FP32 equalization with two to four clusters, whose antennas several lane
groups share.  Accuracy: the RMS errors of z and sigma^2 against 64 bits are those of
the contraction and solve launches, which split a cluster's antennas as far, within a
fifth (the order of the products differs, not the length of the sums).  Edges: fewer
antennas than parts, parts of uneven sizes, clusters of one size and an empty one,
one and two lane groups per warp, parts of lane groups and of one lane (many
subcarriers of small clusters); bounds of test_gpu_parity (FP32)."""
import numpy as np
import pytest

import parity
from oracle import lmmse
from paper_1808_04473_gb300 import synth
from test_gpu_parity import ff  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(ff, p, C, sizes, two_stages):  # noqa: F811
    dev = torch.device("cuda:0")
    plan = ff.ffeq_plan_create(p.B, p.U, C, p.n_sc, p.n_sym, arch=ff.FD, cluster_sizes=sizes)
    nb = ff.ffeq_workspace_size(plan)
    ws = torch.empty(nb, dtype=torch.uint8, device=dev)
    z = torch.empty((p.n_sc, p.n_sym, p.U), dtype=torch.complex64, device=dev)
    s2 = torch.empty((p.n_sc, p.U), device=dev)
    info = torch.full((p.n_sc, C), -1, dtype=torch.int32, device=dev)
    H, y = torch.from_numpy(p.H).to(dev), torch.from_numpy(p.y).to(dev)
    if two_stages:
        ff.ffeq_local_preprocess(plan, H, y, ws, nb)
        ff.ffeq_fuse_equalize(plan, ws, nb, p.N0, p.Es, z, s2, None, info)
    else:
        ff.ffeq_equalize(plan, H, y, p.N0, p.Es, z, s2, None, info, ws, nb)
    torch.cuda.synchronize()
    assert (info == 0).all()
    return z.cpu().numpy(), s2.cpu().numpy()


@pytest.mark.parametrize("B,U,C,n_sc,n_sym", [(64, 4, 2, 200, 1), (256, 8, 2, 100, 2), (256, 11, 2, 320, 14),
                                              (1024, 4, 2, 60, 1), (2000, 3, 2, 60, 1), (255, 15, 3, 320, 14),
                                              (510, 6, 3, 100, 5), (512, 16, 4, 60, 4), (256, 30, 4, 60, 7),
                                              (126, 8, 2, 320, 14), (120, 12, 2, 320, 8), (180, 7, 3, 320, 2),
                                              (248, 16, 4, 320, 3)])
def test_error_is_that_of_the_two_launches(ff, B, U, C, n_sc, n_sym):  # noqa: F811
    p = synth.make_problem(B, U, C, n_sc, n_sym, snr_db=10.0, bits=4, seed=B + U)
    o = lmmse.equalize_fd(p.H, p.y, float(np.float32(p.N0)), p.Es, C, "unbiased")
    err = lambda a, b: np.linalg.norm(a - b) / np.linalg.norm(b)  # noqa: E731
    one, two = _run(ff, p, C, None, False), _run(ff, p, C, None, True)
    for i, k in enumerate(("z", "sigma2")):
        assert err(one[i], o[k]) <= 1.2 * err(two[i], o[k]), (k, err(one[i], o[k]), err(two[i], o[k]))


@pytest.mark.parametrize("B,U,C,n_sc,n_sym,sizes", [(4, 2, 2, 3, 1, None), (6, 16, 2, 320, 14, None),
                                                    (9, 9, 3, 2, 8, None), (34, 5, 3, 5, 9, [1, 0, 33]),
                                                    (30, 8, 2, 4, 4, [29, 1]), (20, 24, 4, 3, 5, None),
                                                    (13, 32, 4, 2, 3, [3, 3, 0, 7]), (8, 1, 4, 1, 16, None),
                                                    (6, 5, 2, 310, 2, None), (9, 9, 3, 310, 8, None),
                                                    (34, 5, 3, 310, 9, [1, 0, 33]), (30, 16, 2, 310, 4, [29, 1])])
def test_parts_edges(ff, B, U, C, n_sc, n_sym, sizes):  # noqa: F811
    p = synth.make_problem(B, U, 1, n_sc, n_sym, snr_db=10.0, bits=4, seed=B + 5 * U)
    N0, part = float(np.float32(p.N0)), sizes if sizes else [B // C] * C
    z, s2 = _run(ff, p, C, sizes, False)
    o = lmmse.equalize_fd(p.H, p.y, N0, p.Es, C, "unbiased", cluster_sizes=part)
    off = np.concatenate([[0], np.cumsum(part)])
    kappa = [max(np.linalg.cond(Hk[:, a:b].conj() @ Hk[:, a:b].T + N0 / p.Es * np.eye(U))
                 for a, b in zip(off[:-1], off[1:])) for Hk in p.H.astype(np.complex128)]
    tol = np.maximum(1e-5, 2.0 * 2.0 ** -22 * np.array(kappa))
    parity.check("z", z, o["z"], tol)
    parity.check("sigma2", s2, o["sigma2"], tol)
