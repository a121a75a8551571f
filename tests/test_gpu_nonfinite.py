"""Infinite and very large values in images: beam-starved pixels reach the
library as infinities, and a residual norm or a backprojection that holds one
is infinite, not NaN."""

import numpy as np
import pytest
import torch

import oracle
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


# Pixels (v, u) of the image of view 2 that are infinite: one, two along a
# detector column, two along a row, a block, many.
@pytest.mark.parametrize("pixels", [[(30, 34)], [(30, 34), (31, 34)], [(30, 34), (30, 35)],
                                    [(30, 34), (31, 34), (30, 35), (31, 35)],
                                    [(v, u) for v in range(15, 45) for u in range(20, 50)]])
@pytest.mark.parametrize("turn,kind", [(0.3, "whole"), (0.3, "window"), (0.3, "event"), (0.3, "subvoxel"),
                                       (20.0, "whole"), (60.0, "whole")])
def test_backprojection(pixels, turn, kind):
    """A voxel whose footprint takes an infinite pixel by a weight that FP32
    resolves (1e-3) is infinite, one beside a footprint keeps its value, and
    no sum of +inf from one view with finite values is NaN.  The detector holds
    the whole blocks of voxels, so that the terms go by the fast paths."""
    from paper_2609_30166_gb300 import ctrex

    P = _matrices(VIEWS, 1, turn, *DET, 220.0, 200.0)
    c = ctrex.Context()
    c.set_geometry(P, SHAPE, (1.0, 1.0, 1.0), ORG, DET)
    pb = oracle.Problem(P, SHAPE, (1.0, 1.0, 1.0), ORG, DET, 0.5)
    if kind == "window":
        win = np.tile([3, DET[0] - 4, 2, DET[1] - 3], (VIEWS, 1)).astype(np.int32)
        c.set_bp_window(win)
        pb = pb.with_window(win)
    elif kind == "event":
        tau, tv = np.full(SHAPE, 0.5), np.linspace(0, 1, VIEWS)
        tau[:, :9] = 0.3
        c.set_dyrect(_t(tau), _t(tv))
        pb = pb.with_dyrect(_np(_t(tau)), _np(_t(tv)))
    elif kind == "subvoxel":
        c.set_bp_subvoxel(2)
        pb = pb.with_subvoxel(2)
    hot, near = np.zeros((VIEWS, DET[1], DET[0])), np.zeros((VIEWS, DET[1], DET[0]))
    for v, u in pixels:
        hot[2, v, u] = 1.0
        near[2, max(v - 1, 0):v + 2, max(u - 1, 0):u + 2] = 1.0
    rng = np.random.default_rng(2)
    base = _np(_t(rng.uniform(0.5, 1.0, size=hot.shape)))
    _, taken, _ = oracle.backproject(pb, hot)
    _, beside, _ = oracle.backproject(pb, near)
    _, plain, _ = oracle.backproject(pb, np.where(near > 0, 0.0, base))
    assert (taken > 1e-3).any()
    free = beside == 0.0
    # a detector coordinate of ~60 holds 4e-6 in FP32 and moves a mean of
    # values in [0.5, 1] by as much; five views and their scales: 1e-4
    got = _np(c.back_project(_t(np.where(hot > 0, np.inf, base)), normalize=False, accumulate=False))
    assert not np.isnan(got).any() and (got[taken > 1e-3] == np.inf).all()
    assert np.abs(got[free] - plain[free]).max(initial=0.0) <= 1e-4
    # NaN beside +inf reaches the footprints that take it, and nothing else
    r = np.where(hot > 0, np.inf, base)
    r[2, 30, 34] = np.nan
    got = _np(c.back_project(_t(r), normalize=False, accumulate=False))
    assert np.isnan(got).any() and np.abs(got[free] - plain[free]).max(initial=0.0) <= 1e-4
    # finite neighbours whose difference is beyond FP32 (the eight
    # points of a sub-voxel mean are summed first, so an eighth of them there)
    big = np.where(hot > 0, 3e38, -2e38 * (near > 0)) / (8.0 if kind == "subvoxel" else 1.0)
    assert not np.isinf(_np(c.back_project(_t(big), normalize=False, accumulate=False))).any()
    c.close()
