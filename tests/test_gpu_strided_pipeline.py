"""The pipelined strided passes (lines of 256 to 1024 points and 3 * 2^m from
384 to 1536): transforms whose x or y pass takes them, with even and odd row
lengths, a last tile of one column, and tile counts below and above the
persistent grid, against the FP64 oracle.  Tolerance as for every FP32
transform: relative L2 2e-6 (u log2(N) of a Cooley-Tukey transform with
correctly rounded twiddles), 1e-5 of the largest coefficient per element.
"""
import numpy as np
import pytest

import synth
from gpu_helpers import from_dev_c64, rel_l2, stream, sync

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fk():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1805_07801_gb300 import build as b

    b.build()
    import paper_1805_07801_gb300 as m

    return m


# (nx, ny, nz): y pass with rows of 33 or 17 columns (odd), x pass with even rows
@pytest.mark.parametrize("shape", [(128, 256, 64), (256, 128, 64), (128, 512, 64), (512, 64, 128), (16, 1024, 64),
                                   (1024, 16, 32), (1024, 6, 32), (128, 384, 64), (384, 128, 32), (12, 768, 64),
                                   (768, 24, 32), (4, 1536, 64), (1536, 6, 48), (128, 512, 48)])
def test_pipelined_passes_match_oracle(fk, oracle_mod, shape):
    import torch

    f = synth.uniform_pm1(61, 0, shape)
    nx, ny, nz = shape
    plan = fk.fftk_plan_create(nx, ny, nz)
    try:
        x = torch.from_numpy(np.ascontiguousarray(f, dtype=np.float32)).to("cuda:0")
        F = torch.empty((nx, ny, nz // 2 + 1, 2), dtype=torch.float32, device="cuda:0")
        y = torch.empty_like(x)
        for _ in range(2):  # the second call finds the tile counters as the first one left them
            fk.fftk_r2c(plan, x.data_ptr(), F.data_ptr(), 1, stream())
            fk.fftk_c2r(plan, F.data_ptr(), y.data_ptr(), 1, stream())
        fk.fftk_sync(plan, stream())
        sync()
        Fg, yg = from_dev_c64(F), y.cpu().numpy()
    finally:
        fk.fftk_plan_destroy(plan)
    want = oracle_mod.rfft3(f.astype(np.float64))
    assert rel_l2(Fg, want) < 2e-6
    assert np.max(np.abs(Fg - want)) < 1e-5 * np.max(np.abs(want))
    assert rel_l2(yg, f) < 2e-6


@pytest.mark.parametrize("basis", ["SCF", "CSF", "SCC", "SFF"])
@pytest.mark.parametrize("shape", [(128, 256, 64), (256, 128, 64), (128, 512, 64), (512, 64, 128), (8, 1024, 64),
                                   (1024, 16, 32)])
def test_pipelined_sine_cosine_passes_match_oracle(fk, oracle_mod, shape, basis):
    import torch

    f = synth.uniform_pm1(62, 0, shape)
    nx, ny, nz = shape
    plan = fk.fftk_plan_create(nx, ny, nz)
    try:
        x = torch.from_numpy(np.ascontiguousarray(f, dtype=np.float32)).to("cuda:0")
        half = basis[2] == "F"
        F = torch.empty((nx, ny, nz // 2 + 1, 2) if half else (nx, ny, nz), dtype=torch.float32, device="cuda:0")
        y = torch.empty_like(x)
        for _ in range(2):
            fk.fftk_forward(plan, basis, x.data_ptr(), F.data_ptr(), 1, stream())
            fk.fftk_inverse(plan, basis, F.data_ptr(), y.data_ptr(), 1, stream())
        fk.fftk_sync(plan, stream())
        sync()
        Fg = from_dev_c64(F) if half else F.cpu().numpy().astype(np.float64)
        yg = y.cpu().numpy()
    finally:
        fk.fftk_plan_destroy(plan)
    want = oracle_mod.transform3(f.astype(np.float64), basis)
    assert rel_l2(Fg, want) < 2e-6
    assert np.max(np.abs(Fg - want)) < 1e-5 * np.max(np.abs(want))
    assert rel_l2(yg, f) < 2e-6
