"""complex128 groups whose values lie outside the range that fixed point takes as they are (csrc/fixed64.cuh: below 2^-895, denormals,
above 2^962), beside ordinary groups and zeros in the same tile: phase A of an axis with p_0 = 8, whose residue classes do not mix,
each class at its own scale; and whole arrays there, with the pointwise product and in a batch.

Bound: the tight one of the ordinary range, 2^-52 (log2 N + 2 d + 1) (every pass rounds once to FP64; the reference's own error is
smaller); results below 2^-1022 are multiples of 2^-1074, so that a pass may be off by 2^-1075 in each component as well, which later
passes add up: with values of 2^-1050 and more that is at most 2^-20 of them over all passes."""
import numpy as np
import pytest

from oracle import cyclic_model as cm
from oracle import rel_l2
from fftu_inputs import complex_uniform

pytestmark = pytest.mark.gpu

EXPONENTS = [-1050, -930, -896, 0, 961, 985, None, -500]  # of the classes; None: zeros


def bound(shape, e):
    n = int(np.prod(shape))
    return 2.0 ** -20 if e < -1000 else 2.0 ** -52 * (np.log2(n) + 2 * len(shape) + 1)


def at(x, e):
    """x 2^e without overflow on the way."""
    return np.ldexp(x.real, e) + 1j * np.ldexp(x.imag, e)


@pytest.fixture(scope="module")
def fftu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2203_11795_gb300
    return paper_2203_11795_gb300


@pytest.mark.parametrize("shape", [(64, 128), (512, 16), (2048, 2), (64, 2, 64)], ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("schedule", [0, 1], ids=["tile", "strided"])
@pytest.mark.parametrize("inverse", [False, True])
def test_classes_at_their_own_scales(fftu, shape, schedule, inverse):
    import torch
    p = (8,) + (1,) * (len(shape) - 1)
    unit = complex_uniform(951, shape, dtype=np.complex128)
    x = np.zeros(shape, np.complex128)
    for s, e in enumerate(EXPONENTS):
        if e is not None:
            x[s::8] = at(unit[s::8], e)
            unit[s::8] = at(x[s::8], -e)  # what the denormals kept
        else:
            unit[s::8] = 0
    t = torch.from_numpy(x).cuda()
    with fftu.Plan(shape, p, dtype=t.dtype, inverse=inverse, schedule=schedule) as plan:
        y = torch.empty_like(t)
        plan.exec_phase(fftu.FFTU_PHASE_A, t, y)
        plan.exec_phase(fftu.FFTU_PHASE_A, t, t)
        assert torch.equal(t, y)
    ref = cm.phase_a(unit, p, inverse=inverse)
    y, m = y.cpu().numpy(), shape[0] // 8
    for s, e in enumerate(EXPONENTS):
        block = y[s * m:(s + 1) * m]
        if e is None:
            assert not block.any()
        else:
            assert rel_l2(at(block, -e), ref[s * m:(s + 1) * m]) <= bound(shape, e), e


@pytest.mark.parametrize("e", [-1050, -930, 985])
@pytest.mark.parametrize("shape", [(8,), (4096,), (64, 64), (512, 64, 64), (16, 32, 8)], ids=lambda s: "x".join(map(str, s)))
def test_whole_arrays(fftu, shape, e):
    import torch
    x = at(complex_uniform(952, shape, dtype=np.complex128), e)
    unit = at(x, -e)
    t = torch.from_numpy(x).cuda()
    with fftu.Plan(shape, None, dtype=t.dtype) as fwd, fftu.Plan(shape, None, dtype=t.dtype, inverse=True) as inv:
        y = fwd.exec(t).cpu().numpy()
        factor = complex_uniform(953, shape, dtype=np.complex128)
        mul = at(factor, -(e // 2))
        u, tmp, out = torch.from_numpy(mul).cuda(), torch.empty_like(t), torch.empty_like(t)
        fftu.fftu_exec_pointwise(fwd.handle, inv.handle, t.data_ptr(), u.data_ptr(), tmp.data_ptr(), out.data_ptr(),
                                 torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
    ref = np.fft.fftn(unit)
    tol = bound(shape, e)
    assert rel_l2(at(y, -e), ref) <= tol
    spec, left = ref * factor, e - e // 2
    assert rel_l2(at(tmp.cpu().numpy(), -left), spec) <= 2 * tol
    assert rel_l2(at(out.cpu().numpy(), -left), np.fft.ifftn(spec)) <= 3 * tol


@pytest.mark.parametrize("inplace", [False, True])
@pytest.mark.parametrize("longest", [(128, 16), (512, 4)], ids=["tables", "roots"])
def test_batch(fftu, longest, inplace):
    """Jobs of one and several stages; 512-point complex128 axes make the batch read the roots instead of tables.  Every shape
    here fits the tile batch's 256 threads, so that the whole batch runs there."""
    import torch
    shapes, exponents = [longest, (8,), (32, 64, 32), (16, 16), longest, (64, 8)], [985, -930, 0, -1050, -896, 985]
    xs = [at(complex_uniform(960 + i, s, dtype=np.complex128), e) for i, (s, e) in enumerate(zip(shapes, exponents))]
    xs[2][3] = np.nan
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
    for i, (x, o, e) in enumerate(zip(xs, outs, exponents)):
        y = o.cpu().numpy()
        if i == 2:
            assert not np.isfinite(y).any()
        else:
            assert rel_l2(at(y, -e), np.fft.fftn(at(x, -e))) <= bound(x.shape, e)
