"""Infinite and very large values in images: beam-starved pixels reach the
library as infinities, and a residual norm or a backprojection that holds one
is infinite, not NaN."""

import numpy as np
import pytest
import torch


from tests.test_gpu_columns import _matrices, _np, _t

pytestmark = pytest.mark.gpu

VIEWS, DET, SHAPE, ORG = 5, (70, 66), (50, 22, 24), (-11.5, -10.5, -24.5)


def _context(turn):
    from paper_2609_30166_gb300 import _build, ctrex

    _build.build_library()
    c = ctrex.Context()
    P = _matrices(VIEWS, 1, turn, *DET, 96.0, 200.0)
    c.set_geometry(P, SHAPE, (1.0, 1.0, 1.0), ORG, DET)
    return c, P


# turn: by columns, by texture gathers
@pytest.mark.parametrize("turn", [0.3, 60.0])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_norms(turn, dtype):
    c, _ = _context(turn)
    x = torch.zeros(SHAPE, device="cuda")
    for value in (float("inf"), float("-inf"), float("nan")):
        p = torch.ones((VIEWS, DET[1], DET[0]), dtype=dtype, device="cuda")
        p[2, 30, 34] = value  # inside the object's shadow
        _, sums = c.fwd_correct(x, p)
        want = float("nan") if np.isnan(value) else float("inf")
        assert np.array_equal(_np(sums), [want, want], equal_nan=True)
    # each tile's partial fits FP32, their total does not
    p = torch.zeros((VIEWS, DET[1], DET[0]), dtype=dtype, device="cuda")
    p[:, ::32, ::32] = 1.5e19
    want = float((p.double() ** 2).sum())
    assert want > 3.5e38
    _, sums = c.fwd_correct(x, p)
    # one product a tile, rounded to FP32; the residual's pixels beyond the shadow count nothing
    assert abs(float(sums[1]) - want) <= 1e-6 * want and np.isfinite(_np(sums)).all()
    c.close()
