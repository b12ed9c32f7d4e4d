"""On a caller's grid fftu_exec gives the bits of its two phases, whichever passes phase A takes (tile, line, pair, triple and
strided ones, the ring of the fused form), out of place and from an in-place phase A of the same passes."""
import numpy as np
import pytest

from fftu_inputs import complex_uniform

pytestmark = pytest.mark.gpu

CASES = [((256, 256), (8, 8)), ((64, 128, 32), (4, 8, 2)), ((16, 16, 128), (2, 4, 8)), ((2048,), (32,)), ((1024, 64), (4, 4)),
         ((32, 32, 32, 32, 32), (4, 4, 4, 4, 4)), ((4096, 8), (4, 1)), ((128, 128, 512), (2, 2, 8)), ((64, 64, 64), (1, 1, 1))]


@pytest.mark.parametrize("dt", [np.complex64, np.complex128])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c[0])))
@pytest.mark.parametrize("inverse", [False, True])
def test_phases_give_the_bits_of_exec(case, dt, inverse):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2203_11795_gb300 as fftu
    shape, p = case
    x = torch.from_numpy(complex_uniform(990, shape, dtype=dt)).cuda()
    with fftu.Plan(shape, p, dtype=x.dtype, inverse=inverse) as plan:
        y, w, u = plan.exec(x), torch.empty_like(x), x.clone()
        plan.exec_phase(fftu.FFTU_PHASE_A, x, w)
        plan.exec_phase(fftu.FFTU_PHASE_B, None, w)
        assert torch.equal(w, y)
        plan.exec_phase(fftu.FFTU_PHASE_A, u, u)
        plan.exec_phase(fftu.FFTU_PHASE_B, None, u)
        plan.exec(x, x)
        assert torch.equal(u, x)
        plan.check_device_status()
