"""Errors of the FP32 transforms against the FP64 oracle, held to what the same
transforms have with correctly rounded factors and radices 16, 16, 4 (or 2) per
line: no pass may lose accuracy to longer radices or to products of factors.
Bounds: relative L2 errors of such passes on these inputs, forward and round
trip, measured to four digits; the inputs are fixed and the kernels' sums have
one order, so nothing is left to chance.  Lines of 1024 points in two radix-32
stages with rounded factors exceed them by 4 and 8 %.
"""
import numpy as np
import pytest

import synth
from gpu_helpers import from_dev_c64, rel_l2, stream, sync

pytestmark = pytest.mark.gpu

# shape, basis, forward error, round-trip error
CASES = [
    ((1024, 16, 32), "FFF", 1.495e-07, 2.284e-07),
    ((16, 1024, 32), "FFF", 1.493e-07, 2.262e-07),
    ((512, 192, 64), "FFF", 1.685e-07, 2.674e-07),
    ((128, 512, 64), "FFF", 1.716e-07, 2.676e-07),
    ((64, 64, 32), "FFF", 1.413e-07, 2.184e-07),
    ((64, 64, 256), "FFF", 1.611e-07, 2.484e-07),
    ((32, 32, 768), "FFF", 1.524e-07, 2.365e-07),
    ((1024, 16, 32), "SFF", 1.575e-07, 2.413e-07),
    ((512, 256, 64), "SCF", 1.906e-07, 3.001e-07),
    ((256, 512, 64), "CSF", 1.906e-07, 2.996e-07),
]


def errors(fk, oracle_mod, shape, basis):
    import torch

    nx, ny, nz = shape
    f = synth.uniform_pm1(63, 0, shape)
    plan = fk.fftk_plan_create(nx, ny, nz)
    try:
        x = torch.from_numpy(np.ascontiguousarray(f, dtype=np.float32)).to("cuda:0")
        F = torch.empty((nx, ny, nz // 2 + 1, 2), dtype=torch.float32, device="cuda:0")
        y = torch.empty_like(x)
        fk.fftk_forward(plan, basis, x.data_ptr(), F.data_ptr(), 1, stream())
        fk.fftk_inverse(plan, basis, F.data_ptr(), y.data_ptr(), 1, stream())
        sync()
        Fg, yg = from_dev_c64(F), y.cpu().numpy()
    finally:
        fk.fftk_plan_destroy(plan)
    want = oracle_mod.rfft3(f.astype(np.float64)) if basis == "FFF" else oracle_mod.transform3(f.astype(np.float64), basis)
    return rel_l2(Fg, want), rel_l2(yg.astype(np.float64), f.astype(np.float64))


@pytest.mark.parametrize("shape,basis,forward,back", CASES)
def test_error_no_larger_than_with_rounded_short_radices(oracle_mod, shape, basis, forward, back):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1805_07801_gb300 import build as b

    b.build()
    import paper_1805_07801_gb300 as fk

    ef, er = errors(fk, oracle_mod, shape, basis)
    assert ef <= forward and er <= back, (ef, er)
