"""The tile sweep of the solve kernel (users that fill no lane group) at the edges
of its shapes: users at and beside the padded sizes 8, 16, 24 and 32, right-hand
sides at and beside 4, 8 and 16, systems of a subcarrier below, at and above what
one CTA takes at once, and both CTA widths (few and many subcarriers).  Bounds of
test_gpu_parity (FP32)."""
import numpy as np
import pytest

from paper_1808_04473_gb300 import synth
from test_gpu_parity import _bound, _check, _gpu, _oracle, ff  # noqa: F401

pytestmark = pytest.mark.gpu

CASES = [
    # B, U, C, n_sc, n_sym, bits
    (40, 1, 1, 5, 1, 2), (60, 7, 2, 33, 4, 4), (80, 9, 2, 9, 5, 2), (96, 15, 3, 160, 8, 6), (128, 17, 4, 6, 9, 4),
    (160, 23, 5, 3, 16, 8), (192, 24, 4, 200, 14, 4), (256, 24, 16, 4, 1, 2), (200, 25, 8, 155, 8, 4),
    (256, 31, 16, 153, 4, 2), (256, 31, 16, 152, 16, 4), (256, 12, 16, 170, 7, 6), (256, 5, 64, 20, 3, 2),
]


@pytest.mark.parametrize("B,U,C,n_sc,n_sym,bits", CASES)
@pytest.mark.parametrize("arch", [0, 1], ids=["PD", "FD"])
@pytest.mark.parametrize("estimate", [0, 1], ids=["unbiased", "literal"])
def test_tile_edges(ff, B, U, C, n_sc, n_sym, bits, arch, estimate):  # noqa: F811
    p = synth.make_problem(B, U, C, n_sc, n_sym, snr_db=10.0, bits=bits, seed=B + 7 * U + C)
    g = _gpu(ff, p, arch, estimate, llr_bits=bits)
    _check(g, _oracle(p, arch, estimate), p, bits, tol=_bound(p, arch, 0))
    assert (g["info"] == 0).all()


@pytest.mark.parametrize("U", [3, 11, 20, 29])
def test_tile_failed_pivot_is_reported_per_system(ff, U):  # noqa: F811
    """Zero forcing with a user no antenna hears: the pivot index, NaN outputs of that subcarrier alone."""
    p = synth.make_problem(64, U, 2, 40, 3, noiseless=True, seed=U)
    H = p.H.copy()
    H[5, U - 1, :] = 0.0
    for arch in (0, 1):
        g = _gpu(ff, p, arch, 0, H=H, N0=0.0)
        info = g["info"].reshape(40, -1)
        assert (info[5] == U).all() and (np.delete(info, 5, 0) == 0).all()
        assert np.isnan(g["z"][5]).all() and np.isfinite(np.delete(g["z"], 5, 0)).all()
