"""complex128 stages in 64-bit fixed point (csrc/fixed64.cuh) against the FP64 oracle: every first-stage radix
(2, 4, 8), one to four stages, per-axis and grouped phase B, wide magnitude spreads, zeros, and the values that
take the FP64 arithmetic instead (exponents out of the scaled range, infinities, NaN).

Bound: a pass rounds its results to FP64 once (relative 2^-53 at most, its fixed-point error being smaller), there
are at most 2 d + 1 passes, and the oracle's own error is about 2^-53 sqrt(log2 N): 2^-52 log2 N + 2^-52 (2 d + 1)
covers both."""
import numpy as np
import pytest

import oracle
from fftu_inputs import complex_uniform

pytestmark = pytest.mark.gpu

CASES = [((64, 64, 64), (2, 2, 2)), ((8, 128), (2, 8)), ((16, 16), (4, 4)), ((2048,), (4,)), ((4096, 2), (1, 1)),
         ((1024, 32), (32, 4)), ((64, 8, 64), (8, 2, 8)), ((4, 2, 256, 16), (2, 1, 16, 2))]


@pytest.fixture(scope="module")
def fftu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2203_11795_gb300
    return paper_2203_11795_gb300


def make(kind, shape):
    x = complex_uniform(404 + len(shape), shape, dtype=np.complex128)
    e = complex_uniform(405, shape, dtype=np.complex128).real
    if kind == "wide":       # 200 decades of magnitudes
        return x * 10.0 ** (100 * e)
    if kind == "padded":     # exact zeros in most lines, and denormals beside ordinary values
        x = np.where(e > 0.5, x, 0.0)
        x.reshape(-1)[::7] = 5e-310
        return x
    if kind == "huge":       # biased exponents above the scaled range
        return x * 2.0 ** 985
    if kind == "tiny":       # below it
        return x * 2.0 ** -920
    return x


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c[0])))
@pytest.mark.parametrize("kind", ["uniform", "wide", "padded", "huge", "tiny"])
@pytest.mark.parametrize("inverse", [False, True])
def test_fixed_point_stages(fftu, case, kind, inverse):
    import torch
    shape, p = case
    x = make(kind, shape)
    t = torch.from_numpy(x).cuda()
    with fftu.Plan(shape, p, dtype=t.dtype, inverse=inverse) as plan:
        y = plan.exec(t).cpu().numpy()
        plan.exec(t, t)
        assert np.array_equal(t.cpu().numpy(), y)  # in place, the same passes
        plan.check_device_status()
    s = {"huge": 2.0 ** -900, "tiny": 2.0 ** 900}.get(kind, 1.0)  # keeps the comparison's own squares finite
    ref = oracle.fftn(x * s, inverse=inverse)
    err = oracle.rel_l2(y * s, ref)
    print(f"{shape} {kind} {'inverse' if inverse else 'forward'}: rel L2 {err:.2e}")
    assert err <= 2.0 ** -52 * (np.log2(x.size) + 2 * len(shape) + 1)


@pytest.mark.parametrize("case", CASES[:3], ids=lambda c: "x".join(map(str, c[0])))
@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_not_finite(fftu, case, value):
    """One infinite or NaN input reaches every output, as in FP64 arithmetic."""
    import torch
    shape, p = case
    x = make("uniform", shape)
    x.reshape(-1)[x.size // 3] = value
    t = torch.from_numpy(x).cuda()
    with fftu.Plan(shape, p, dtype=t.dtype) as plan:
        y = plan.exec(t).cpu().numpy()
    assert not np.isfinite(y).any()


def test_zero_array(fftu):
    import torch
    t = torch.zeros((32, 32), dtype=torch.complex128, device="cuda")
    with fftu.Plan((32, 32), (4, 4), dtype=t.dtype) as plan:
        assert not plan.exec(t).abs().any()
