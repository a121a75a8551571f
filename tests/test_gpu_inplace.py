"""Corrections written over the measured images."""

import pytest
import torch

from tests.test_gpu_columns import _matrices

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("turn", [0.3, 60.0])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_fwd_correct_in_place(turn, dtype):
    """fwd_correct(x, p, r=p): a pixel is read before it is written, and both
    norms are those of p as it was."""
    from paper_2609_30166_gb300 import _build, ctrex

    _build.build_library()
    views, det, shape = 5, (45, 66), (40, 22, 24)
    c = ctrex.Context()
    c.set_geometry(_matrices(views, 1, turn, *det, 96.0, 200.0), shape, (1.0, 1.0, 1.0), (-11.5, -10.5, -19.5), det)
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.rand(shape, generator=g, device="cuda")
    p = (2.0 + torch.rand((views, det[1], det[0]), generator=g, device="cuda")).to(dtype)
    want, sums = c.fwd_correct(x, p)
    got, inplace = c.fwd_correct(x, p, r=p)
    assert got.data_ptr() == p.data_ptr() and torch.equal(got, want) and torch.equal(inplace, sums)
    c.close()
