"""One context used from two streams at once: its calls share the column stores
and the adjoint's scatter volume, so each has to wait for the one before it.

Either call alone is the reference: the projector and the backprojector give
the same bits again, the adjoint and the motion gradient add in another order
(1e-5 relative L2, the operators' contract)."""

import numpy as np
import pytest
import torch

from tests.helpers import rel_l2
from tests.test_gpu_columns import _matrices, _np, _t

pytestmark = pytest.mark.gpu

VIEWS, DET, SHAPE = 40, (160, 160), (128, 120, 112)


def _context(motion):
    from paper_2609_30166_gb300 import _build, ctrex

    _build.build_library()
    c = ctrex.Context()
    c.set_geometry(_matrices(VIEWS, 1, 0.3, *DET, 200.0, 400.0), SHAPE, (0.5, 0.5, 0.5), (-27.75, -29.75, -31.75), DET)
    if motion:
        theta = np.zeros((VIEWS, 15))
        theta[:, 6:] = np.eye(3).ravel()
        coef = np.random.default_rng(5).uniform(-1, 1, (8, 8, 8, 3))
        c.set_motion(_t(theta), _t(coef), _t(np.linspace(0.2, 1.0, VIEWS)), 0.5)
    return c


def _calls(c, motion):
    g = torch.Generator(device="cuda").manual_seed(7)
    xs = [torch.rand(SHAPE, generator=g, device="cuda") for _ in range(2)]
    ys = [torch.rand((VIEWS, DET[1], DET[0]), generator=g, device="cuda") for _ in range(2)]
    ops = {"adjoint": lambda k: c.adjoint_project(ys[k]), "forward": lambda k: c.fwd_project(xs[k]),
           "backproject": lambda k: c.back_project(ys[k], normalize=False, accumulate=False)}
    if motion:
        ops["gradient"] = lambda k: c.motion_grad(xs[k], ys[k])[1]
    return ops


@pytest.mark.parametrize("motion", [False, True])
@pytest.mark.parametrize("pair", [("adjoint", "adjoint"), ("forward", "forward"), ("backproject", "backproject"),
                                  ("adjoint", "forward"), ("gradient", "forward"), ("gradient", "gradient")])
def test_two_streams(pair, motion):
    if "gradient" in pair and not motion or pair == ("forward", "forward") and motion:
        pytest.skip("no gradient without motion; the projector with motion reads its texture atlas")
    c = _context(motion)
    ops = _calls(c, motion)
    want = [_np(ops[name](k)) for k, name in enumerate(pair)]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    for _ in range(5):
        got = []
        for k, name in enumerate(pair):
            with torch.cuda.stream(streams[k]):
                got.append(ops[name](k))
        torch.cuda.synchronize()
        for a, b, name in zip(got, want, pair):
            if name in ("adjoint", "gradient"):
                assert rel_l2(_np(a), b) <= 1e-5
            else:
                assert np.array_equal(_np(a), b)
    c.close()
