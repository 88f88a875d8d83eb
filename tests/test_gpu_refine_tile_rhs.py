"""The one-step refinement tiles at the ends of their symbol widths (4, 8 and 16), for
each padded user count, one warp and several per system.  Bound of
test_gpu_refine_tile."""
import pytest

from test_gpu_refine import ff  # noqa: F401
from test_gpu_refine_tile import test_one_step_edges as _one_step

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_sym", [4, 5, 7, 8, 9])
@pytest.mark.parametrize("B,U,C,arch", [(32, 6, 2, 1), (98, 8, 1, 0), (98, 13, 1, 0), (48, 16, 3, 1), (98, 20, 1, 0),
                                        (64, 32, 2, 1)])
def test_symbol_widths(ff, B, U, C, arch, n_sym):  # noqa: F811
    _one_step(ff, B, U, C, 4, n_sym, None, arch, 2 if arch == 0 else 0, 0)
