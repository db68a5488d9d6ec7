"""Calls of a few rows, which take kernels of their own: the role-routed linear map of at
most 192 rows (weights as the M operand, reduction split over a cluster), at the edges
of its row paddings (16, 32, 64, 128, 192), with and without a split, ragged column
tiles, one kind of row or both."""
import numpy as np
import pytest

from paper_2601_21927_gb300 import inputs
from tests.test_gpu_routed import _check, _roles, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 16, 17, 32, 33, 64, 65, 128, 129, 191, 192, 193])
def test_routed_linear_row_paddings(T):
    """Reductions of 3 steps (no split) and 16 steps (split by up to 4); 160 columns end
    inside a 128-row weight tile and inside a part."""
    for d_in, seed in ((192, 31), (1024, 32)):
        r = _run(_roles(T, T + seed), d_in, [96, 32, 32], [False, True, True], seed=seed,
                 cache_rows=2 * T + 5, x_pad=64)
        _check(r)


@pytest.mark.parametrize("role", [inputs.ROLE_CURR, inputs.ROLE_NEXUS, None])
@pytest.mark.parametrize("T,d_in,cols", [(7, 4096, [4096, 1024, 1024]), (40, 3584, [3584]),
                                         (190, 2048, [2048, 512, 512]), (130, 2112, [4640])])
def test_routed_linear_projection_widths(role, T, d_in, cols):
    roles = _roles(T, T) if role is None else np.full(T, role, np.uint8)
    r = _run(roles, d_in, cols, [False] + [True] * (len(cols) - 1), seed=41, cache_rows=T + 9)
    _check(r)
