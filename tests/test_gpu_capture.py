"""Operators inside a stream capture.  A capturing stream can neither allocate
nor wait for another stream's work, so there the adjoint and the motion
gradient use the caller's buffers and what set_motion allocated, as their first
call on a context may be the captured one; the projector and the backprojector
read what earlier calls have laid out."""

import ctypes

import numpy as np
import pytest
import torch

from tests.helpers import rel_l2
from tests.test_gpu_columns import _matrices, _np, _t

pytestmark = pytest.mark.gpu

VIEWS, DET, SHAPE, VOX, ORG = 6, (64, 64), (50, 36, 32), (1.0, 1.0, 1.0), (-15.5, -17.5, -24.5)


def _context(motion=False, shape=SHAPE, det=DET):
    from paper_2609_30166_gb300 import _build, ctrex

    _build.build_library()
    c = ctrex.Context()
    c.set_geometry(_matrices(VIEWS, 1, 0.3, *det, 96.0, 200.0), shape, VOX, ORG, det)
    if motion:
        theta = np.zeros((VIEWS, 15))
        theta[:, 6:] = np.eye(3).ravel()
        c.set_motion(_t(theta), _t(np.random.default_rng(5).uniform(-1, 1, (8, 8, 8, 3))),
                     _t(np.linspace(0.2, 1.0, VIEWS)), 0.5)
    return c


def _capture(call):
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = call()
    return graph, out


def _images(det=DET):
    return torch.rand((VIEWS, det[1], det[0]), generator=torch.Generator(device="cuda").manual_seed(3), device="cuda")


@pytest.mark.parametrize("motion", [False, True])
def test_first_adjoint_and_gradient(motion):
    c, y = _context(motion), _images()
    x = torch.rand(SHAPE, generator=torch.Generator(device="cuda").manual_seed(4), device="cuda")
    vol = torch.zeros(SHAPE, device="cuda")
    gt, gc = torch.zeros((VIEWS, 15), device="cuda"), torch.zeros((8, 8, 8, 3), device="cuda")

    def call():
        c.adjoint_project(y, vol=vol)
        if motion:
            c.motion_grad(x, y, grad_theta=gt, grad_coef=gc)

    graph, _ = _capture(call)
    vol.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert rel_l2(_np(vol), _np(c.adjoint_project(y))) <= 1e-5
    if motion:
        want_t, want_c = c.motion_grad(x, y)
        assert rel_l2(_np(gt), _np(want_t)) <= 1e-4 and rel_l2(_np(gc), _np(want_c)) <= 1e-4
        # replayed beside an eager call on another stream
        for _ in range(5):
            vol.zero_()
            torch.cuda.synchronize()
            graph.replay()
            with torch.cuda.stream(torch.cuda.Stream()):
                other = c.adjoint_project(2.0 * y)
            torch.cuda.synchronize()
            assert rel_l2(2.0 * _np(vol), _np(other)) <= 1e-5
    c.close()


def test_projectors_after_a_first_call():
    c, y = _context(), _images()
    x = torch.rand(SHAPE, generator=torch.Generator(device="cuda").manual_seed(4), device="cuda")
    p, b = c.fwd_project(x), c.back_project(y, normalize=False, accumulate=False)
    (graph, (q, d)) = _capture(lambda: (c.fwd_project(x), c.back_project(y, normalize=False, accumulate=False)))
    x.mul_(2.0)
    y.mul_(2.0)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(q, 2.0 * p) and torch.equal(d, 2.0 * b)
    c.close()


def test_layout_is_not_left_to_the_replay():
    """A store that would have to be laid out anew is not taken in a capture:
    its border would be written by the replay only, and an eager call before
    that would read another layout's values.  (Nor are texture atlases, so the
    captured call fails.)"""
    P = _matrices(VIEWS, 1, 0.3, *DET, 40.0, 200.0)  # the object is truncated
    c = _context(shape=(100, 72, 64), det=(128, 128))
    c.back_project(_images((128, 128)))
    c.fwd_project(torch.rand((100, 72, 64), device="cuda"))
    c.set_geometry(P, SHAPE, VOX, ORG, DET)
    fresh = _context()
    fresh.set_geometry(P, SHAPE, VOX, ORG, DET)
    y, x = _images(), torch.rand(SHAPE, device="cuda")
    b, p = torch.zeros(SHAPE, device="cuda"), torch.zeros_like(y)
    torch.cuda.synchronize()
    cuda, graph, stream = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(), torch.cuda.Stream()
    for call in (lambda k: k.back_project(y, vol=b, normalize=False, accumulate=False),
                 lambda k: k.fwd_project(x, proj=p)):
        with torch.cuda.stream(stream):
            handle = ctypes.c_void_p(stream.cuda_stream)
            assert cuda.cuStreamBeginCapture_v2(handle, 2) == 0  # relaxed: allocations are allowed
            try:
                call(c)
            except RuntimeError:
                pass
            cuda.cuStreamEndCapture(handle, ctypes.byref(graph))
        got = _np(call(c))
        assert np.array_equal(got, _np(call(fresh)))
    c.close()
    fresh.close()
