"""The column kernels (*_column*.cu) at the edges of their tiles
and of the rules that choose them, against the FP64 oracle.

Both choices compute the same operator, so every case holds to the projector's
contract, 1e-5 relative L2 (FP32 storage): detectors of 31, 32 and 33 rows and
of widths beside a multiple of 4, volumes of 1 to 130 slices (a thread's 2 or 4
voxels, 64- and 128-slice blocks that overlap), detectors turned to either side
of the rules' limits, a detector smaller than the object's shadow (blocks of
voxels inside, across and outside its edge), and a source inside the volume;
and each other forward model on both sides of the rule, by columns and by
texture gathers.
"""

import math

import numpy as np
import pytest
import torch

import oracle
from paper_2609_30166_gb300 import inputs
from tests.helpers import rel_l2

pytestmark = pytest.mark.gpu

TOL32 = 1e-5

# (nx, ny, nz), (nu, nv), views, sub-angles, in-plane turn of the detector (deg), detector width (mm), SOD (mm)
CASES = [
    ((33, 20, 64), (45, 31), 7, 1, 0.4, 96.0, 200.0),
    ((32, 33, 65), (48, 32), 6, 2, 0.0, 96.0, 200.0),
    ((19, 37, 130), (31, 33), 5, 1, -0.3, 96.0, 200.0),
    ((40, 8, 127), (130, 96), 3, 1, 1.0, 96.0, 200.0),
    ((41, 29, 1), (50, 64), 5, 1, 0.2, 96.0, 200.0),
    ((1, 40, 40), (50, 40), 5, 1, 0.2, 96.0, 200.0),
    ((24, 24, 66), (36, 64), 5, 1, 28.0, 96.0, 200.0),   # below both limits
    ((24, 24, 40), (36, 64), 5, 1, 40.0, 96.0, 200.0),   # forward by columns, backprojection by gathers
    ((24, 24, 40), (36, 64), 5, 1, 55.0, 96.0, 200.0),   # both by gathers
    ((48, 40, 90), (33, 40), 9, 1, 0.5, 40.0, 200.0),    # truncated: part of the object off the detector
    ((24, 24, 40), (48, 48), 6, 1, 0.0, 96.0, 10.0),     # source inside the volume
    ((96, 90, 70), (24, 32), 6, 1, 0.0, 96.0, 200.0),    # pixel steps of several voxels
    ((16, 16, 40), (96, 160), 6, 1, 0.0, 96.0, 200.0),   # voxel steps of several pixels
]


def _matrices(views, sub, turn, nu, nv, width, sod):
    rng = np.random.default_rng(5)
    t, pitch = math.radians(turn), width / nu
    P = np.zeros((views, sub, 3, 4))
    for v in range(views):
        du, dv = rng.uniform(-1.5, 1.5, 2)
        for s in range(sub):
            R = inputs.rot_z(0.3 + 2 * math.pi * (v + 0.2 * s) / views)
            u, w = R @ np.array([0.0, pitch, 0.0]), np.array([0.0, 0.0, pitch])
            ctr = R @ np.array([200.0, 0.0, 0.0]) + du * u + dv * w
            P[v, s] = inputs.cone_matrix(R @ np.array([-sod, 0.0, 0.0]), ctr, math.cos(t) * u + math.sin(t) * w,
                                         math.cos(t) * w - math.sin(t) * u, nu, nv)
    return P


def _t(a, dtype=torch.float32):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64).to(dtype).cuda().contiguous()


def _np(t):
    return t.detach().double().cpu().numpy()


@pytest.mark.parametrize("n,det,views,sub,turn,width,sod", CASES)
def test_columns_match_oracle(n, det, views, sub, turn, width, sod):
    from paper_2609_30166_gb300 import _build, ctrex

    _build.build_library()
    (nx, ny, nz), (nu, nv) = n, det
    P = _matrices(views, sub, turn, nu, nv, width, sod)
    pitch = 32.0 / max(nx, ny, 1.3 * nz)
    vox = (pitch, pitch, 1.3 * pitch)
    org = tuple(-0.5 * (m - 1) * v for m, v in zip(n, vox))
    rng = np.random.default_rng(9)
    x = rng.uniform(0.2, 1.0, size=(nz, ny, nx))
    pb = oracle.Problem(P, (nz, ny, nx), vox, org, det, 0.5)
    c = ctrex.Context()
    c.set_geometry(P, (nz, ny, nx), vox, org, det)
    ref, rs = oracle.forward(pb, _np(_t(x)))
    rows = torch.empty(ref.shape, device="cuda")
    assert rel_l2(_np(c.fwd_project(_t(x), rowsum=rows)), ref) <= TOL32
    assert rel_l2(_np(rows), rs) <= TOL32
    # BF16 volume, FP32 result; a second pass over the kept store
    x16 = _t(x, torch.bfloat16)
    assert rel_l2(_np(c.fwd_project(x16, out_dtype=torch.float32)), oracle.forward(pb, _np(x16))[0]) <= TOL32
    # smooth images: an FP32 detector coordinate resolves noise to ~1e-4 only
    iu, iv = np.meshgrid(np.arange(nu), np.arange(nv))
    r = np.stack([np.cos(0.11 * iu + k) + np.sin(0.07 * iv * (k + 1)) + 2.5 for k in range(views)])
    w = rng.uniform(0.5, 1.0, size=x.shape)
    want, b, _ = oracle.backproject(pb, _np(_t(r)), w=_np(_t(w)), alpha=0.7, x=_np(_t(x)))
    got = c.back_project(_t(r), vol=_t(x), w=_t(w), alpha=0.7)
    assert rel_l2(_np(got), want) <= TOL32
    assert rel_l2(_np(c.back_project(_t(r), normalize=False, accumulate=False)), b) <= TOL32
    # a view list: out of order, fewer images than the kept store holds
    vi = np.arange(views)[::-2].astype(np.int32).copy()
    _, b, _ = oracle.backproject(pb, _np(_t(r[vi])), views=vi)
    assert rel_l2(_np(c.back_project(_t(r[vi]), normalize=False, accumulate=False, view_idx=vi)), b) <= TOL32
    c.close()


@pytest.mark.parametrize("model", ["event", "joseph", "roi", "cylinder"])
@pytest.mark.parametrize("turn,tall", [(0.4, False), (44.0, True), (60.0, False)])
def test_models_match_oracle(model, turn, tall):
    """turn: columns, columns near the limit, gathers.  tall: steep rays over a
    short detector distance, so that the Joseph projector's principal axis is
    z on some of them and x or y on others."""
    from paper_2609_30166_gb300 import _build, ctrex

    _build.build_library()
    n, det, views = (22, 27, 41), (37, 66), 6
    P = _matrices(views, 1, turn, det[0], det[1], 250.0 if tall else 80.0, 60.0 if tall else 200.0)
    vox = (1.0, 0.9, 0.8)
    org = tuple(-0.5 * (m - 1) * v for m, v in zip(n, vox))
    rng = np.random.default_rng(4)
    shape = n[::-1]
    c = ctrex.Context()
    if model == "cylinder":
        shape = (41, 30, 17)  # slices, sectors, rings
        args = dict(n_r=17, n_phi=30, n_z=41, dr=0.8, dz=0.8)
        c.set_geometry_cylinder(P, det=det, **args)
        pb = oracle.cylinder_problem(P, det=det, **args)
    else:
        c.set_geometry(P, shape, vox, org, det)
        pb = oracle.Problem(P, shape, vox, org, det, 0.5)
    if model == "event":
        # regions that change early, late, never and (NaN) at once, and a gradual front
        tau = np.full(shape, 2.0)
        tau[:, :13] = 0.1 + 0.8 * np.linspace(0, 1, shape[0])[:, None, None]
        tau[5:9, 20:23, 3:9] = np.nan
        tv = np.linspace(0, 1, views)
        c.set_dyrect(_t(tau), _t(tv))
        pb = pb.with_dyrect(_np(_t(tau)), _np(_t(tv)))
        shape = (2,) + shape
    elif model == "joseph":
        c.set_projector("joseph")
        pb = pb.with_joseph()
    elif model == "roi":
        roi = ((19, 21, 23), (0.3, 0.3, 0.35), (-2.5, -1.0, 0.7))
        c.set_roi(*roi)
        pb = pb.with_roi(*roi)
        shape = (c.vol_shape[0],)
    x = rng.uniform(0.2, 1.0, size=shape)
    rows = torch.empty((views, det[1], det[0]), device="cuda")
    for dt in (torch.float32, torch.bfloat16):
        ref, rs = oracle.forward(pb, _np(_t(x, dt)))
        got = c.fwd_project(_t(x, dt), rowsum=rows, out_dtype=torch.float32)
        assert rel_l2(_np(got), ref) <= TOL32
        assert rel_l2(_np(rows), rs) <= TOL32
    c.close()


@pytest.mark.parametrize("n,det,views,sub,turn", [
    ((37, 22, 65), (45, 33), 5, 1, 0.4),    # rows of a detector column
    ((32, 64, 31), (130, 40), 3, 2, 2.0),
    ((20, 31, 96), (33, 64), 5, 1, 30.0),   # patches
    ((41, 24, 30), (31, 50), 5, 1, 70.0),
    ((1, 40, 33), (40, 40), 5, 1, 0.0),
    ((64, 64, 64), (12, 5), 1, 1, 0.0),     # few rays: in place
])
@pytest.mark.parametrize("motion", [False, True])
def test_adjoint_matches_oracle(n, det, views, sub, turn, motion):
    from paper_2609_30166_gb300 import _build, ctrex

    _build.build_library()
    P = _matrices(views, sub, turn, det[0], det[1], 96.0, 200.0)
    pitch = 30.0 / max(n)
    vox, shape = (pitch, 0.9 * pitch, 1.1 * pitch), n[::-1]
    org = tuple(-0.5 * (m - 1) * v for m, v in zip(n, vox))
    pb = oracle.Problem(P, shape, vox, org, det, 0.5)
    c = ctrex.Context()
    c.set_geometry(P, shape, vox, org, det)
    rng = np.random.default_rng(21)
    if motion:
        theta = np.zeros((views, 15))
        theta[:, :6] = rng.uniform(-0.02, 0.02, (views, 6))
        theta[:, 6:] = np.eye(3).ravel() + rng.uniform(-0.01, 0.01, (views, 9))
        coef, sv = rng.uniform(-1, 1, (8, 8, 8, 3)) * 1.5 * pitch, np.linspace(0.2, 1.0, views)
        theta, coef, sv = (_np(_t(a)) for a in (theta, coef, sv))  # as the GPU sees them
        pb = pb.with_motion(theta, coef, sv, margin=0.5)
        c.set_motion(_t(theta), _t(coef), _t(sv), 0.5)
    y = rng.uniform(0.5, 1.5, size=(views, det[1], det[0]))
    x0 = rng.uniform(size=shape)
    want = oracle.adjoint(pb, _np(_t(y)))
    got = _np(c.adjoint_project(_t(y), vol=_t(x0))) - _np(_t(x0))  # accumulates
    assert rel_l2(got, want) <= TOL32
    vi = np.arange(views)[::-2].astype(np.int32).copy()
    want = oracle.adjoint(pb, _np(_t(y[vi])), views=vi)
    assert rel_l2(_np(c.adjoint_project(_t(y[vi]), view_idx=vi)), want) <= TOL32
    if motion:
        x = rng.uniform(0.2, 1.0, size=shape)
        assert rel_l2(_np(c.fwd_project(_t(x))), oracle.forward(pb, _np(_t(x)))[0]) <= TOL32
    c.close()


# Motion by runs of samples in one spline cell: a step short enough for runs in
# every operator, in the adjoint and the gradient only, and in the full gradient
# but not in the pose's.  Poses that carry rays beyond the spline's domain (its
# coordinate is clamped there), steps along a cell's faces, sub-angles.
# Projector and adjoint: the contract.  Gradient: positions hold about 2e-6
# voxels, so some 1e-5 of the samples lie on the other side of a voxel face,
# where this volume's gradient turns by a few percent, in a sum that cancels to
# about 1 % of its terms: 1e-4.
@pytest.mark.parametrize("n,det,views,sub,turn,step,shift", [
    ((30, 41, 35), (37, 22), 4, 1, 0.4, 0.1, 0.0),
    ((33, 32, 30), (21, 33), 3, 2, 30.0, 0.08, 6.0),   # beyond the clamp on one side
    ((30, 30, 50), (9, 40), 5, 1, 0.0, 0.17, -3.0),    # 35 samples a cell: not in the projector
    ((5, 40, 40), (20, 12), 4, 1, 2.0, 0.02, 1.0),     # cells of one voxel
    ((30, 30, 30), (31, 5), 3, 1, 0.0, 0.1, 0.0),
])
def test_motion_runs_match_oracle(n, det, views, sub, turn, step, shift):
    from paper_2609_30166_gb300 import _build, ctrex

    _build.build_library()
    P = _matrices(views, sub, turn, det[0], det[1], 60.0, 200.0)
    pitch = 30.0 / max(n)
    vox, shape = (pitch, 0.95 * pitch, 1.05 * pitch), n[::-1]
    org = tuple(-0.5 * (m - 1) * v for m, v in zip(n, vox))
    rng = np.random.default_rng(33)
    theta = np.zeros((views, 15))
    theta[:, :6] = rng.uniform(-0.03, 0.03, (views, 6))
    theta[:, 3] += shift * pitch
    theta[:, 6:] = np.eye(3).ravel() + rng.uniform(-0.01, 0.01, (views, 9))
    coef, sv = rng.uniform(-1, 1, (8, 8, 8, 3)) * 0.05 * max(n) * pitch, np.linspace(0.2, 1.0, views)
    theta, coef, sv = (_np(_t(a)) for a in (theta, coef, sv))  # as the GPU sees them
    pb = oracle.Problem(P, shape, vox, org, det, step).with_motion(theta, coef, sv, margin=0.5)
    c = ctrex.Context()
    c.set_geometry(P, shape, vox, org, det, step_vox=step)
    c.set_motion(_t(theta), _t(coef), _t(sv), 0.5)
    axes = [(np.arange(m) + 1.0) * (m - np.arange(m)) / (m + 1.0) ** 2 for m in shape]
    x = 64.0 * axes[0][:, None, None] * axes[1][:, None] * axes[2]
    y = rng.uniform(0.5, 1.5, size=(views, det[1], det[0]))
    y[:, ::3, 1::2] = 0.0  # rays without weight
    x, y = _np(_t(x)), _np(_t(y))
    rows = torch.empty((views, det[1], det[0]), device="cuda")
    ref, rs = oracle.forward(pb, x)
    assert rel_l2(_np(c.fwd_project(_t(x), rowsum=rows)), ref) <= TOL32
    assert rel_l2(_np(rows), rs) <= TOL32
    assert rel_l2(_np(c.adjoint_project(_t(y))), oracle.adjoint(pb, y)) <= TOL32
    gt, gc = oracle.motion_grad(pb, x, y)
    got_t, got_c = c.motion_grad(_t(x), _t(y))
    assert rel_l2(_np(got_t), gt) <= 1e-4 and rel_l2(_np(got_c), gc) <= 1e-4
    assert rel_l2(_np(c.motion_grad(_t(x), _t(y), want_coef=False)[0]), gt) <= 1e-4
    vi = np.arange(views)[::-2].astype(np.int32).copy()
    ref, _ = oracle.forward(pb, x, views=vi)
    assert rel_l2(_np(c.fwd_project(_t(x), view_idx=vi)), ref) <= TOL32
    gt, gc = oracle.motion_grad(pb, x, y[vi], views=vi)
    got_t, got_c = c.motion_grad(_t(x), _t(y[vi]), view_idx=vi)
    assert rel_l2(_np(got_t), gt) <= 1e-4 and rel_l2(_np(got_c), gc) <= 1e-4
    c.close()


# Backprojection where every view holds the whole volume, in lists of 32 terms:
# one term, lists with a remainder, sub-angles, an image repeated; thin volumes
# (blocks of slices beyond the last one) and a detector that the volume nearly
# fills, or is just too large for.
@pytest.mark.parametrize("n,det,views,sub,turn,width", [
    ((9, 11, 130), (48, 90), 33, 1, 0.4, 96.0),
    ((17, 8, 64), (40, 44), 35, 2, 0.0, 96.0),
    ((8, 8, 5), (33, 31), 1, 1, -2.0, 96.0),
    ((30, 30, 128), (41, 61), 32, 1, 1.0, 83.0),
    ((30, 30, 30), (64, 64), 20, 4, 0.0, 74.0),
    ((1, 31, 70), (50, 60), 7, 1, 0.3, 96.0),
])
def test_flat_backprojection_matches_oracle(n, det, views, sub, turn, width):
    from paper_2609_30166_gb300 import _build, ctrex

    _build.build_library()
    P = _matrices(views, sub, turn, det[0], det[1], width, 200.0)
    pitch = 30.0 / max(n)
    vox, shape = (pitch, 0.9 * pitch, pitch), n[::-1]
    org = tuple(-0.5 * (m - 1) * v for m, v in zip(n, vox))
    c = ctrex.Context()
    c.set_geometry(P, shape, vox, org, det)
    pb = oracle.Problem(P, shape, vox, org, det, 0.5)
    rng = np.random.default_rng(17)
    x, w = rng.uniform(0.2, 1.0, size=shape), rng.uniform(0.5, 1.0, size=shape)
    iu, iv = np.meshgrid(np.arange(det[0]), np.arange(det[1]))
    r = np.stack([np.cos(0.11 * iu + k) + np.sin(0.07 * iv * (k % 5 + 1)) + 2.5 for k in range(views)])
    want, b, _ = oracle.backproject(pb, _np(_t(r)), w=_np(_t(w)), alpha=0.7, x=_np(_t(x)))
    assert rel_l2(_np(c.back_project(_t(r), vol=_t(x), w=_t(w), alpha=0.7)), want) <= TOL32
    assert rel_l2(_np(c.back_project(_t(r), normalize=False, accumulate=False)), b) <= TOL32
    vi = np.concatenate([np.arange(views)[::-3], [0, 0]]).astype(np.int32)
    _, b, _ = oracle.backproject(pb, _np(_t(r[vi])), views=vi)
    assert rel_l2(_np(c.back_project(_t(r[vi]), normalize=False, accumulate=False, view_idx=vi)), b) <= TOL32
    # 16-bit images and volume: one rounding of the result (2^-9)
    r16 = _t(r, torch.bfloat16)
    want, _, _ = oracle.backproject(pb, _np(r16), alpha=0.7)
    got = c.back_project(r16, alpha=0.7, vol_dtype=torch.bfloat16)
    assert rel_l2(_np(got), want) <= 2.0 ** -8
    c.close()


# |p|^2 of fwd_correct: FP32 in tiles of 32 x 4 pixels (a butterfly over each
# row of 32, then row by row), FP64 over the tiles; the last sum's order is
# free: 1e-13.
@pytest.mark.parametrize("det,dtype", [((45, 31), torch.float32), ((64, 33), torch.bfloat16), ((31, 66), torch.float32)])
def test_correction_norm_by_tiles(det, dtype):
    from paper_2609_30166_gb300 import _build, ctrex

    _build.build_library()
    nu, nv = det
    views, shape = 5, (40, 22, 24)
    c = ctrex.Context()
    c.set_geometry(_matrices(views, 1, 0.2, nu, nv, 96.0, 200.0), shape, (1.0, 1.0, 1.0), (-11.5, -10.5, -19.5), det)
    rng = np.random.default_rng(3)
    p = _t(rng.uniform(0.0, 2.0, size=(views, nv, nu)), dtype)
    x = _t(rng.uniform(size=shape))
    sums = torch.empty(2, dtype=torch.float64, device="cuda")
    vi = np.array([4, 1, 3], dtype=np.int32)
    for k, idx in ((views, None), (3, vi)):
        c.fwd_correct(x, p[:k].contiguous(), sums=sums, view_idx=idx)
        q = np.zeros((k, -(-nv // 4) * 4, -(-nu // 32) * 32), dtype=np.float32)
        q[:, :nv, :nu] = p[:k].float().cpu().numpy()
        v = (q * q).reshape(k, -1, 4, q.shape[2] // 32, 32)
        for off in (16, 8, 4, 2, 1):
            v = v[..., :off] + v[..., off:2 * off]
        t = np.zeros(v.shape[:2] + v.shape[3:4], dtype=np.float32)
        for r in range(4):
            t = t + v[:, :, r, :, 0]
        want = t.astype(np.float64).sum()
        assert abs(sums[1].item() - want) <= 1e-13 * want
    c.close()



# Detectors whose 8-row bands are more than a launch holds: 300 x 262140 pixels,
# of which the object's shadow takes the middle rows (rays are formed relative
# to the detector's middle in FP32).  Reference: the same rays on a detector of
# those rows alone.
@pytest.mark.parametrize("motion,turn", [(True, 0.0), (False, 20.0)])
def test_adjoint_of_tall_detector(motion, turn):
    from paper_2609_30166_gb300 import _build, ctrex

    _build.build_library()
    nu, nv, shadow, shape = 300, 262140, 100, (20, 18, 16)
    vox, org = (1.0, 1.0, 1.0), tuple(-0.5 * (m - 1) for m in shape[::-1])
    P = _matrices(1, 1, turn, nu, shadow, 96.0, 200.0)
    first = (nv - shadow) // 2
    rng = np.random.default_rng(8)
    pb = oracle.Problem(P, shape, vox, org, (nu, shadow), 0.5)
    c = ctrex.Context()
    shift = np.array([[1.0, 0.0, 0.0], [0.0, 1.0, first], [0.0, 0.0, 1.0]])
    c.set_geometry(shift @ P, shape, vox, org, (nu, nv))  # the same rows, and more on both sides
    if motion:
        theta = np.zeros((1, 15))
        theta[:, :6] = rng.uniform(-0.02, 0.02, (1, 6))
        theta[:, 6:] = np.eye(3).ravel()
        coef, sv = rng.uniform(-1, 1, (8, 8, 8, 3)), np.ones(1)
        theta, coef = _np(_t(theta)), _np(_t(coef))
        pb = pb.with_motion(theta, coef, sv, margin=0.5)
        c.set_motion(_t(theta), _t(coef), _t(sv), 0.5)
    y = torch.zeros((1, nv, nu), device="cuda")
    rows = y[:, first:first + shadow]
    rows.copy_(_t(rng.uniform(0.5, 1.5, size=(1, shadow, nu))))
    want = oracle.adjoint(pb, _np(rows))
    assert rel_l2(_np(c.adjoint_project(y)), want) <= TOL32
    c.close()


# Views whose time scale is 0 see no deformation, whatever its coefficients
# are, sample by sample and by runs.
@pytest.mark.parametrize("step", [0.5, 0.08])
def test_views_without_deformation(step):
    from paper_2609_30166_gb300 import _build, ctrex

    _build.build_library()
    n, det, views = (30, 41, 35), (37, 22), 4
    P = _matrices(views, 1, 0.4, det[0], det[1], 60.0, 200.0)
    vox, shape = (0.7, 0.7, 0.7), n[::-1]
    org = tuple(-0.5 * (m - 1) * v for m, v in zip(n, vox))
    rng = np.random.default_rng(12)
    theta = np.zeros((views, 15))
    theta[:, :6] = rng.uniform(-0.03, 0.03, (views, 6))
    theta[:, 6:] = np.eye(3).ravel()
    theta = _np(_t(theta))
    coef = np.full((8, 8, 8, 3), np.inf)
    coef[::2] = np.nan
    pb = oracle.Problem(P, shape, vox, org, det, step).with_motion(theta, None, None, margin=0.5)
    c = ctrex.Context()
    c.set_geometry(P, shape, vox, org, det, step_vox=step)
    c.set_motion(_t(theta), _t(coef), _t(np.array([0.0, 1.0, 0.0, 1.0])), 0.5)
    x, y = rng.uniform(0.2, 1.0, size=shape), rng.uniform(0.5, 1.5, size=(2, det[1], det[0]))
    vi = np.array([0, 2], dtype=np.int32)
    assert rel_l2(_np(c.fwd_project(_t(x), view_idx=vi)), oracle.forward(pb, _np(_t(x)), views=vi)[0]) <= TOL32
    assert rel_l2(_np(c.adjoint_project(_t(y), view_idx=vi)), oracle.adjoint(pb, _np(_t(y)), views=vi)) <= TOL32
    c.close()


# Detectors on both sides of the lean at which a model and a storage type
# change from columns to gathers (static BF16 about 8 degrees, Joseph about 17),
# and rows of which columns waste too many lanes on the cylinder (33).
@pytest.mark.parametrize("model,turn,nv", [("static", 6.0, 60), ("static", 11.0, 60), ("joseph", 14.0, 60),
                                           ("joseph", 21.0, 60), ("cylinder", 0.3, 33), ("cylinder", 30.0, 60)])
def test_lean_limits_of_models(model, turn, nv):
    from paper_2609_30166_gb300 import _build, ctrex

    _build.build_library()
    n, det, views = (22, 27, 41), (37, nv), 5
    P = _matrices(views, 1, turn, det[0], det[1], 80.0, 200.0)
    shape = n[::-1]
    c = ctrex.Context()
    if model == "cylinder":
        shape = (41, 30, 17)  # slices, sectors, rings
        args = dict(n_r=17, n_phi=30, n_z=41, dr=0.8, dz=0.8)
        c.set_geometry_cylinder(P, det=det, **args)
        pb = oracle.cylinder_problem(P, det=det, **args)
    else:
        vox = (1.0, 0.9, 0.8)
        org = tuple(-0.5 * (m - 1) * v for m, v in zip(n, vox))
        c.set_geometry(P, shape, vox, org, det)
        pb = oracle.Problem(P, shape, vox, org, det, 0.5)
    if model == "joseph":
        c.set_projector("joseph")
        pb = pb.with_joseph()
    x = np.random.default_rng(4).uniform(0.2, 1.0, size=shape)
    for dt in (torch.float32, torch.bfloat16):
        ref, _ = oracle.forward(pb, _np(_t(x, dt)))
        assert rel_l2(_np(c.fwd_project(_t(x, dt), out_dtype=torch.float32)), ref) <= TOL32
    c.close()


# Motion by the pose alone: straight displaced rays, in every operator, and
# the gradient with respect to the pose with and without a deformation beside
# it; tolerances as in test_motion_runs_match_oracle.
@pytest.mark.parametrize("n,det,views,sub,turn,step", [
    ((30, 41, 35), (37, 22), 4, 1, 0.4, 0.5),
    ((33, 32, 70), (21, 33), 3, 2, 30.0, 0.08),
    ((5, 40, 8), (70, 5), 5, 1, 0.0, 0.5),
    ((64, 64, 64), (12, 5), 1, 1, 60.0, 0.5),   # few rays
])
def test_pose_only_matches_oracle(n, det, views, sub, turn, step):
    from paper_2609_30166_gb300 import _build, ctrex

    _build.build_library()
    P = _matrices(views, sub, turn, det[0], det[1], 60.0, 200.0)
    pitch = 30.0 / max(n)
    vox, shape = (pitch, 0.95 * pitch, 1.05 * pitch), n[::-1]
    org = tuple(-0.5 * (m - 1) * v for m, v in zip(n, vox))
    rng = np.random.default_rng(34)
    theta = np.zeros((views, 15))
    theta[:, :6] = rng.uniform(-0.03, 0.03, (views, 6))
    theta[:, 6:] = np.eye(3).ravel() + rng.uniform(-0.01, 0.01, (views, 9))
    coef = rng.uniform(-1, 1, (8, 8, 8, 3)) * 0.05 * max(n) * pitch
    theta, coef = (_np(_t(a)) for a in (theta, coef))  # as the GPU sees them
    c = ctrex.Context()
    c.set_geometry(P, shape, vox, org, det, step_vox=step)
    axes = [(np.arange(m) + 1.0) * (m - np.arange(m)) / (m + 1.0) ** 2 for m in shape]
    x = _np(_t(64.0 * axes[0][:, None, None] * axes[1][:, None] * axes[2]))
    y = _np(_t(rng.uniform(0.5, 1.5, size=(views, det[1], det[0]))))
    plain = oracle.Problem(P, shape, vox, org, det, step)
    for co, sv in ((None, None), (coef, np.ones(views))):
        pb = plain.with_motion(theta, co, sv, margin=0.5)
        c.set_motion(_t(theta), None if co is None else _t(co), None if sv is None else _t(sv), 0.5)
        rows = torch.empty((views, det[1], det[0]), device="cuda")
        ref, rs = oracle.forward(pb, x)
        assert rel_l2(_np(c.fwd_project(_t(x), rowsum=rows)), ref) <= TOL32
        assert rel_l2(_np(rows), rs) <= TOL32
        assert rel_l2(_np(c.adjoint_project(_t(y))), oracle.adjoint(pb, y)) <= TOL32
        gt, _ = oracle.motion_grad(pb, x, y)
        assert rel_l2(_np(c.motion_grad(_t(x), _t(y), want_coef=False)[0]), gt) <= 1e-4
    c.close()


# The adjoint's patches for a few rows, and (64 slices, fine pixels, turned)
# in place by the pose alone and with a deformation.
@pytest.mark.parametrize("n,det,views,turn", [((37, 22, 9), (90, 12), 5, 0.4), ((37, 22, 9), (90, 17), 5, 0.4),
                                              ((64, 60, 64), (190, 190), 12, 60.0)])
@pytest.mark.parametrize("motion", ["none", "pose", "full"])
def test_adjoint_of_few_rows_and_turned(n, det, views, turn, motion):
    from paper_2609_30166_gb300 import _build, ctrex

    _build.build_library()
    P = _matrices(views, 1, turn, det[0], det[1], 60.0, 200.0)
    pitch = 30.0 / max(n)
    vox, shape = (pitch, 0.95 * pitch, 1.05 * pitch), n[::-1]
    org = tuple(-0.5 * (m - 1) * v for m, v in zip(n, vox))
    rng = np.random.default_rng(35)
    pb = oracle.Problem(P, shape, vox, org, det, 0.5)
    c = ctrex.Context()
    c.set_geometry(P, shape, vox, org, det)
    if motion != "none":
        theta = np.zeros((views, 15))
        theta[:, :6] = rng.uniform(-0.03, 0.03, (views, 6))
        theta[:, 6:] = np.eye(3).ravel()
        theta = _np(_t(theta))
        coef = _np(_t(rng.uniform(-1, 1, (8, 8, 8, 3)) * pitch)) if motion == "full" else None
        sv = np.ones(views) if motion == "full" else None
        pb = pb.with_motion(theta, coef, sv, margin=0.5)
        c.set_motion(_t(theta), None if coef is None else _t(coef), None if sv is None else _t(sv), 0.5)
    y = _np(_t(rng.uniform(0.5, 1.5, size=(views, det[1], det[0]))))
    assert rel_l2(_np(c.adjoint_project(_t(y))), oracle.adjoint(pb, y)) <= TOL32
    c.close()


# Backprojection by columns in every model, at heights whose blocks of 64 or 128
# slices fit, overlap or (a tiny volume) reach beyond the last one; by FP32 and
# 16-bit images, a view list, sub-angles.
@pytest.mark.parametrize("model", ["static", "window", "event", "cylinder", "roi", "subvoxel"])
@pytest.mark.parametrize("nz,sub,width", [(64, 4, 220.0), (100, 1, 220.0), (127, 1, 70.0), (150, 2, 220.0), (250, 1, 90.0),
                                          (5, 1, 220.0)])
def test_backprojection_blocks_match_oracle(model, nz, sub, width):
    from paper_2609_30166_gb300 import _build, ctrex

    _build.build_library()
    nx, ny, det, views = 11, 9, (60, 76), 5
    P = _matrices(views, sub, 0.3, *det, width, 200.0)
    pitch = 30.0 / max(nz, 20)
    shape, vox = (nz, ny, nx), (pitch, pitch, pitch)
    org = tuple(-0.5 * (m - 1) * pitch for m in (nx, ny, nz))
    rng = np.random.default_rng(11)
    c = ctrex.Context()
    if model == "cylinder":
        shape, args = (nz, ny, 6), dict(n_r=6, n_phi=ny, n_z=nz, dr=pitch, dz=pitch)
        c.set_geometry_cylinder(P, det=det, **args)
        pb = oracle.cylinder_problem(P, det=det, **args)
    else:
        c.set_geometry(P, shape, vox, org, det)
        pb = oracle.Problem(P, shape, vox, org, det, 0.5)
    if model == "window":
        win = np.stack([[3 + v, det[0] - 5, 4, det[1] - 9 + v] for v in range(views)]).astype(np.int32)
        c.set_bp_window(win)
        pb = pb.with_window(win)
    elif model == "event":
        tau, tv = rng.uniform(0.0, 1.0, size=shape), np.linspace(0, 1, views)
        c.set_dyrect(_t(tau), _t(tv))
        pb = pb.with_dyrect(_np(_t(tau)), _np(_t(tv)))
    elif model == "roi":
        roi = ((max(nz // 2, 1), 7, 8), (0.5 * pitch,) * 3, (-1.75 * pitch, -1.5 * pitch, -0.25 * (max(nz // 2, 1) - 1) * pitch))
        c.set_roi(*roi)
        pb = pb.with_roi(*roi)
    elif model == "subvoxel":
        c.set_bp_subvoxel(2)
        pb = pb.with_subvoxel(2)
    iu, iv = np.meshgrid(np.arange(det[0]), np.arange(det[1]))
    r = np.stack([np.cos(0.11 * iu + k) + np.sin(0.07 * iv * (k + 1)) + 2.5 for k in range(views)])
    x = rng.uniform(0.2, 1.0, size=c.vol_shape)
    want, b, _ = oracle.backproject(pb, _np(_t(r)), alpha=0.7, x=_np(_t(x)))
    assert rel_l2(_np(c.back_project(_t(r), vol=_t(x), alpha=0.7)), want) <= TOL32
    r16 = _t(r, torch.bfloat16)
    _, b, _ = oracle.backproject(pb, _np(r16))
    assert rel_l2(_np(c.back_project(r16, normalize=False, accumulate=False)), b) <= TOL32
    vi = np.array([4, 1], dtype=np.int32)
    _, b, _ = oracle.backproject(pb, _np(_t(r[vi])), views=vi)
    assert rel_l2(_np(c.back_project(_t(r[vi]), normalize=False, accumulate=False, view_idx=vi)), b) <= TOL32
    c.close()
