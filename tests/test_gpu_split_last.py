"""Split-precision plans whose sub-FFTs end in a CUDA-core stage of radix 2, 4 or 8 (csrc/generic_tiles.cuh,
stockham_last) against the oracle: strided and contiguous axes, runs shorter than a warp, in place, lines longer than a
tile, both directions.  Tolerance: the library's own for complex64 (relative L2 1e-5 log2 N)."""
import math

import numpy as np
import pytest

import oracle
from fftu_inputs import complex_uniform

pytestmark = pytest.mark.gpu

# sub-FFT lengths 32 (16 x 2), 64 (16 x 4), 128 (16 x 8), 512 (16 x 16 x 2) and 2048 (16 x 16 x 8)
CASES = [((64, 64), (2, 2)), ((32, 4, 2), (1, 2, 1)), ((256, 32, 8), (4, 1, 2)), ((2, 1024), (1, 8)), ((1024, 2), (2, 1)),
         ((16384, 4), (8, 2)), ((4, 16384), (2, 8)), ((128, 16, 64), (1, 1, 1))]


@pytest.mark.parametrize("precision", [1, 2], ids=["bf16", "fp16"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c[0])))
@pytest.mark.parametrize("inverse", [False, True])
def test_split_last_stage(case, precision, inverse):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2203_11795_gb300 as fftu
    shape, p = case
    x = complex_uniform(910 + len(shape), shape, dtype=np.complex64)
    t = torch.from_numpy(x).cuda()
    with fftu.Plan(shape, p, dtype=t.dtype, inverse=inverse, precision=precision) as plan:
        y = plan.exec(t).cpu().numpy()
        assert np.array_equal(t.cpu().numpy(), x)
        if max(shape) <= 8192:  # longer lines are refused in place
            plan.exec(t, t)
            assert np.array_equal(t.cpu().numpy(), y)
        plan.check_device_status()
    ref = oracle.fftn(x.astype(np.complex128), inverse=inverse)
    assert oracle.rel_l2(y, ref) <= 1e-5 * math.log2(x.size)
