"""complex128 on data that a few values dominate, whose later stages do not grow (csrc/fixed64.cuh: block floating point):
an impulse, a few values, a point source over a background, a plane wave, a strong mean; in groups of up to 4096 points of the
tile passes (whole axes, two axes in one tile, phase A) and of the strided passes.

Bound: a pass holds a group's inputs to a unit of at most 2^-57 of the largest, so 2^-56.5 sqrt(n) of the results'
norm for n = 2^12 points, 2^-50.5; all later roundings of the pass together are kept below as much: 2^-50.  At
most d passes on the library's grid, d and one on a caller's.  The reference is numpy's FFT in FP64, whose own error is about
2^-53 sqrt(log2 N): twice that."""
import numpy as np
import pytest

from oracle import rel_l2
from fftu_inputs import complex_uniform

pytestmark = pytest.mark.gpu

AUTO, GENERIC = 0, 1
CASES = [((4096,), None, AUTO), ((2, 4096), None, AUTO), ((4096, 2), None, AUTO), ((512, 64, 64), None, AUTO),
         ((1024, 16), None, AUTO), ((16, 8, 8, 64), None, AUTO), ((4096, 8), (2, 1), AUTO), ((2, 16, 4096), (1, 4, 1), AUTO),
         ((4096, 2), (1, 1), GENERIC), ((8, 2048), (2, 1), GENERIC)]


def data(kind, shape):
    x = complex_uniform(930 + len(shape), shape, dtype=np.complex128)
    at = tuple(5 * n // 7 for n in shape)
    if kind == "normal":
        z = np.random.default_rng(931).standard_normal((2, *shape))
        return z[0] + 1j * z[1]
    if kind == "wave":
        phase = sum(2 * np.pi * ((3 * l + 5) % n) / n * np.arange(n).reshape([-1 if k == l else 1 for k in range(len(shape))])
                    for l, n in enumerate(shape))
        return np.exp(1j * phase)
    if kind == "mean":
        return 1 + 1e-3 * x
    if kind == "few":
        y = np.zeros(shape, np.complex128)
        y.reshape(-1)[:: max(1, x.size // 4) + 1] = x.reshape(-1)[:: max(1, x.size // 4) + 1]
        return y
    background = {"impulse": 0.0, "source3": 1e-3, "source2": 1e-2, "source1": 1e-1}[kind]
    y = background * x
    y[at] = 1.0 + 0.3j
    return y


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c[0])) + ("g" if c[2] else "p" if c[1] else ""))
@pytest.mark.parametrize("kind", ["impulse", "few", "source3", "source2", "source1", "wave", "mean", "normal"])
def test_dominated_by_few_values(case, kind):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2203_11795_gb300 as fftu
    shape, p, schedule = case
    x = data(kind, shape)
    bound = (len(shape) + (p is not None)) * 2.0 ** -50 + 2.0 ** -52 * np.sqrt(np.log2(x.size))
    t = torch.from_numpy(x).cuda()
    for inverse in (False, True):
        with fftu.Plan(shape, p, dtype=t.dtype, inverse=inverse, schedule=schedule) as plan:
            y = plan.exec(t).cpu().numpy()
        err = rel_l2(y, (np.fft.ifftn if inverse else np.fft.fftn)(x))
        print(f"{shape} {p} {kind} {'inverse' if inverse else 'forward'}: {err:.2e}, bound {bound:.2e}")
        assert err <= bound
