"""Tile passes (csrc/tile_pass.cu) against the oracle and the CPU model of Algorithm 2.3: whole axes (default grid) and
phase A (a caller's grid), at the edges of their range: one to four digits per axis, groups of one to three axes, the
smallest and largest tiles, strided and contiguous, in and out of place, with the pointwise product.

Tolerances: the library's own (relative L2 1e-5 log2 N for complex64, 1e-12 for complex128)."""
import math

import numpy as np
import pytest

import oracle
from oracle import cyclic_model as cm
from fftu_inputs import complex_uniform

pytestmark = pytest.mark.gpu

WHOLE = [(2,), (16,), (32,), (4096,), (4, 2), (2, 2, 2), (16, 16), (8, 4096), (1024, 4), (1024, 1024), (64, 64, 64),
         (32, 2, 128), (128, 32, 256), (1, 64, 1, 512), (16, 8, 4, 4, 2), (32, 32, 32, 32), (512, 2, 16)]
GRIDS = [((256, 256), (8, 8)), ((1024, 64), (4, 4)), ((64, 128, 32), (4, 8, 2)), ((512, 32, 32), (16, 4, 1)),
         ((8, 1024), (2, 16)), ((4096, 8), (4, 1)), ((16, 16, 128), (2, 4, 8)), ((2048,), (32,)), ((128, 4, 16), (8, 2, 4))]


def tol(dt, n):
    return 1e-12 if dt == np.complex128 else 1e-5 * max(1.0, math.log2(n))


def shape_id(s):
    return "x".join(map(str, s))


@pytest.fixture(scope="module")
def fftu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2203_11795_gb300
    return paper_2203_11795_gb300


@pytest.mark.parametrize("dt", [np.complex64, np.complex128])
@pytest.mark.parametrize("shape", WHOLE, ids=shape_id)
@pytest.mark.parametrize("inverse", [False, True])
def test_whole_axes(fftu, shape, dt, inverse):
    import torch
    x = complex_uniform(71 + len(shape), shape, dtype=dt)
    t = torch.from_numpy(x).cuda()
    with fftu.Plan(shape, None, dtype=t.dtype, inverse=inverse) as plan:
        y = plan.exec(t).cpu().numpy()
        assert np.array_equal(t.cpu().numpy(), x)
        if dt == np.complex64 or max(shape) <= 4096:  # longer complex128 lines are refused in place
            plan.exec(t, t)
            assert np.array_equal(t.cpu().numpy(), y)
        plan.check_device_status()
    assert oracle.rel_l2(y, oracle.fftn(x.astype(np.complex128), inverse=inverse)) <= tol(dt, x.size)


@pytest.mark.parametrize("dt", [np.complex64, np.complex128])
@pytest.mark.parametrize("case", GRIDS, ids=lambda c: shape_id(c[0]))
@pytest.mark.parametrize("inverse", [False, True])
def test_phase_a(fftu, case, dt, inverse):
    """Phase A alone = Supersteps 0 + 1 of the model, in and out of place; then the whole transform."""
    import torch
    shape, p = case
    x = complex_uniform(72 + len(shape), shape, dtype=dt)
    t = torch.from_numpy(x).cuda()
    with fftu.Plan(shape, p, dtype=t.dtype, inverse=inverse) as plan:
        w = torch.empty_like(t)
        plan.exec_phase(fftu.FFTU_PHASE_A, t, w)
        u = t.clone()
        plan.exec_phase(fftu.FFTU_PHASE_A, u, u)
        y = plan.exec(t).cpu().numpy()
        plan.exec_phase(fftu.FFTU_PHASE_B, None, w.clone())
        plan.check_device_status()
    ref = cm.phase_a(x.astype(np.complex128), p, inverse=inverse)
    assert oracle.rel_l2(w.cpu().numpy(), ref) <= tol(dt, x.size)
    assert oracle.rel_l2(u.cpu().numpy(), ref) <= tol(dt, x.size)
    assert oracle.rel_l2(y, oracle.fftn(x.astype(np.complex128), inverse=inverse)) <= tol(dt, x.size)


@pytest.mark.parametrize("dt", [np.complex64, np.complex128])
@pytest.mark.parametrize("shape", [(16,), (64, 64), (32, 16, 64)], ids=shape_id)
def test_pointwise(fftu, shape, dt):
    import torch
    x, m = (complex_uniform(s, shape, dtype=dt) for s in (91, 92))
    t, u = torch.from_numpy(x).cuda(), torch.from_numpy(m).cuda()
    tmp, out = torch.empty_like(t), torch.empty_like(t)
    with fftu.Plan(shape, None, dtype=t.dtype) as fwd, fftu.Plan(shape, None, dtype=t.dtype, inverse=True) as inv:
        fftu.fftu_exec_pointwise(fwd.handle, inv.handle, t.data_ptr(), u.data_ptr(), tmp.data_ptr(), out.data_ptr(),
                                 torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
    spec = oracle.fftn(x.astype(np.complex128)) * m
    assert oracle.rel_l2(tmp.cpu().numpy(), spec) <= tol(dt, x.size)
    assert oracle.rel_l2(out.cpu().numpy(), oracle.fftn(spec, inverse=True)) <= tol(dt, x.size)


@pytest.mark.parametrize("kind", ["huge", "tiny", "nan"])
def test_values_out_of_the_fixed_point_range(fftu, kind):
    """complex128 tiles that run again in FP64, whole axes in place and phase A."""
    import torch
    shape = (64, 16, 32)
    x = complex_uniform(93, shape, dtype=np.complex128) * {"huge": 2.0 ** 985, "tiny": 2.0 ** -930, "nan": 1.0}[kind]
    if kind == "nan":
        x[5, 3, 7] = np.nan
    s = {"huge": 2.0 ** -900, "tiny": 2.0 ** 900, "nan": 1.0}[kind]
    t = torch.from_numpy(x).cuda()
    with fftu.Plan(shape, None, dtype=t.dtype) as whole, fftu.Plan(shape, (4, 2, 4), dtype=t.dtype) as grid:
        z = grid.exec(t).cpu().numpy()
        whole.exec(t, t)
        y = t.cpu().numpy()
    if kind == "nan":
        assert not np.isfinite(y).any() and not np.isfinite(z).any()
        return
    ref = oracle.fftn(x * s)
    assert oracle.rel_l2(y * s, ref) <= 1e-12 and oracle.rel_l2(z * s, ref) <= 1e-12


@pytest.mark.parametrize("dt", [np.complex64, np.complex128])
@pytest.mark.parametrize("inplace", [False, True])
def test_batch_of_tile_passes(fftu, dt, inplace):
    """One launch over transforms of one to three whole-axis passes, tiny to several thousand points an axis; in
    complex128 one of them holds values that take FP64 arithmetic."""
    import torch
    shapes = [(32, 64, 128), (16,), (2, 2), (4096,), (8, 1024), (128, 32, 32), (64, 4, 4, 16), (1, 256, 2)]
    xs = [complex_uniform(700 + i, s, dtype=dt) for i, s in enumerate(shapes)]
    scale = [1.0] * len(xs)
    if dt == np.complex128:
        xs[5], scale[5] = xs[5] * 2.0 ** 985, 2.0 ** -900
    ts = [torch.from_numpy(x).cuda() for x in xs]
    outs = ts if inplace else [torch.empty_like(t) for t in ts]
    plans = [fftu.Plan(s, None, dtype=t.dtype) for s, t in zip(shapes, ts)]
    b = fftu.fftu_batch_create([p.handle for p in plans])
    fftu.fftu_batch_exec(b, [t.data_ptr() for t in ts], [o.data_ptr() for o in outs],
                         torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    fftu.fftu_batch_check_status(b)
    fftu.fftu_batch_destroy(b)
    for p in plans:
        p.close()
    for x, o, s in zip(xs, outs, scale):
        assert oracle.rel_l2(o.cpu().numpy() * s, oracle.fftn(x.astype(np.complex128) * s)) <= tol(dt, x.size)


@pytest.mark.parametrize("dt", [np.complex64, np.complex128])
@pytest.mark.parametrize("longest", [512, 1024], ids=lambda n: f"longest{n}")
def test_batch_tables(fftu, dt, longest):
    """Batches on both sides of the twiddle tables' largest size (512-point complex64 axes have them, 1024-point ones and
    512-point complex128 ones take the roots), with passes of one to three stages and without twiddles."""
    import torch
    shapes = [(longest, 4), (2, longest), (8, 8, 8), (16, 16, 16), (64, 32, 128), (256, 64), (2,)]
    xs = [complex_uniform(810 + i, s, dtype=dt) for i, s in enumerate(shapes)]
    ts = [torch.from_numpy(x).cuda() for x in xs]
    outs = [torch.empty_like(t) for t in ts]
    plans = [fftu.Plan(s, None, dtype=t.dtype, inverse=True) for s, t in zip(shapes, ts)]
    b = fftu.fftu_batch_create([p.handle for p in plans])
    for _ in range(2):
        fftu.fftu_batch_exec(b, [t.data_ptr() for t in ts], [o.data_ptr() for o in outs],
                             torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    fftu.fftu_batch_check_status(b)
    fftu.fftu_batch_destroy(b)
    for p in plans:
        p.close()
    for x, o in zip(xs, outs):
        assert oracle.rel_l2(o.cpu().numpy(), oracle.fftn(x.astype(np.complex128), inverse=True)) <= tol(dt, x.size)


@pytest.mark.parametrize("shape", [(512, 64, 64), (8, 64, 64, 64)], ids=shape_id)
def test_two_axes_of_64_complex128(fftu, shape):
    """Contiguous planes of 64 x 64 in one tile, in and out of place; one plane takes FP64 arithmetic."""
    import torch
    x = complex_uniform(820, shape, dtype=np.complex128)
    x[1] *= 2.0 ** -980
    t = torch.from_numpy(x).cuda()
    with fftu.Plan(shape, None, dtype=t.dtype) as plan:
        y = plan.exec(t)
        assert torch.equal(t, torch.from_numpy(x).cuda())
        plan.exec(t, t)
        assert torch.equal(t, y)
        plan.check_device_status()
    assert oracle.rel_l2(y.cpu().numpy(), oracle.fftn(x)) <= tol(np.complex128, x.size)
