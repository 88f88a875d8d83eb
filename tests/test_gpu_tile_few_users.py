"""The solve tiles where padding users are left out: pivots past the last user's trip
are not swept and the epilogue walks the users alone where they fill at most half of
the tile.  Users at and beside the ends of a trip (4 pivots with 8 and 16 padded users,
12 with 24, 8 with 32), outputs that fill no CTA, both architectures, refinement (the
estimates and inverses that the sweep leaves) and a failing last pivot.  Bounds of
test_gpu_parity and test_gpu_refine."""
import numpy as np
import pytest

from paper_1808_04473_gb300 import synth
from test_gpu_parity import _bound, _check, _gpu, _oracle, ff  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("U", [1, 2, 3, 4, 5, 9, 12, 13, 17, 21, 25, 27])
@pytest.mark.parametrize("arch", [0, 1], ids=["PD", "FD"])
@pytest.mark.parametrize("n_sc,n_sym,bits", [(85, 14, 8), (3, 1, 2), (157, 5, 6)])
def test_trips_and_outputs(ff, U, arch, n_sc, n_sym, bits):  # noqa: F811
    p = synth.make_problem(90, U, 3, n_sc, n_sym, snr_db=10.0, bits=bits, seed=U + n_sc)
    g = _gpu(ff, p, arch, 0, llr_bits=bits, precision=2)   # BF16x3: the solve kernel for both architectures
    _check(g, _oracle(p, arch, 0), p, bits, tol=_bound(p, arch, 2))
    assert (g["info"] == 0).all()


@pytest.mark.parametrize("U", [3, 4, 12, 20])
@pytest.mark.parametrize("arch", [0, 1], ids=["PD", "FD"])
def test_refined(ff, U, arch):  # noqa: F811
    p = synth.make_problem(96, U, 2, 20, 6, snr_db=12.0, bits=4, seed=U)
    dev = torch.device("cuda:0")
    out = ff.equalize(torch.from_numpy(p.H).to(dev), torch.from_numpy(p.y).to(dev), p.N0, p.Es, 2, arch=arch, llr_bits=4,
                      precision=2, refine=1)
    g = {k: v.cpu().numpy() for k, v in out.items()}
    _check(g, _oracle(p, arch, 0), p, 4, tol=_bound(p, arch, 0))


@pytest.mark.parametrize("U", [1, 4, 12, 21, 27])
def test_last_pivot_fails(ff, U):  # noqa: F811
    p = synth.make_problem(64, U, 2, 40, 3, noiseless=True, seed=U)
    H = p.H.copy()
    H[7, U - 1, :] = 0.0
    for arch in (0, 1):
        g = _gpu(ff, p, arch, 0, H=H, N0=0.0, precision=2)
        info = g["info"].reshape(40, -1)
        assert (info[7] == U).all() and (np.delete(info, 7, 0) == 0).all()
        assert np.isnan(g["z"][7]).all() and np.isfinite(np.delete(g["z"], 7, 0)).all()
