"""Every variant of the pipelined strided pass against the FP64 oracle: line
length, row parity (even rows as whole boxes, odd ones as two tensors), Fourier,
sine and cosine, forward and inverse, always with more tiles than resident CTAs,
so that a CTA refills its staging buffer under a transform and reuses its exchange
buffer, and with two calls in a row on one plan (the tile counters).  The dispatch
rule is restated here, so that a shape that fell back to the general pass fails.
Tolerance as for every FP32 transform: relative L2 2e-6, 1e-5 of the largest
coefficient per element.
"""
import numpy as np
import pytest

import synth
from gpu_helpers import from_dev_c64, rel_l2, stream, sync

pytestmark = pytest.mark.gpu

CTAS_PER_SM = {256: 4, 384: 2, 512: 2, 768: 1, 1024: 1, 1536: 1}
TURNS = {256: 3, 384: 2, 512: 2, 768: 1, 1024: 1, 1536: 1}  # tiles per resident CTA

# shape, basis, the passes aimed at (axis 0: x, 1: y)
CASES = [
    ((1024, 256, 32), "FFF", (0, 1)),  # y 256 odd, x 1024 even
    ((256, 1024, 64), "FFF", (0, 1)),  # y 1024 odd, x 256 even
    ((384, 512, 48), "FFF", (0, 1)),   # y 512 odd, x 384 even
    ((512, 384, 64), "FFF", (0, 1)),   # y 384 odd, x 512 even
    ((96, 768, 32), "FFF", (1,)),      # odd
    ((768, 96, 64), "FFF", (0,)),      # even
    ((64, 1536, 32), "FFF", (1,)),     # odd
    ((1536, 48, 64), "FFF", (0,)),     # even
    ((256, 1024, 64), "SFF", (0,)),    # 256 even: its inverse
    ((256, 1024, 64), "CFF", (0,)),
    ((512, 512, 64), "SCF", (0, 1)),   # y odd, x even
    ((512, 512, 64), "CSF", (0, 1)),
    ((512, 512, 64), "CCS", (0, 1)),   # both even
    ((512, 512, 64), "SSC", (0, 1)),
    ((1024, 256, 32), "SFF", (0,)),    # even
    ((1024, 256, 32), "CFF", (0,)),
    ((128, 1024, 32), "SCF", (1,)),    # odd
    ((128, 1024, 32), "CSF", (1,)),
    ((256, 1024, 32), "CSC", (1,)),    # even
    ((256, 1024, 32), "SCS", (1,)),
]


def takes_the_pipeline(shape, basis, axis, sms):
    nx, ny, nz = shape
    qy = nz // 2 + 1 if basis[2] == "F" else nz // 2
    L, P, Q = (nx, 1, ny * qy) if axis == 0 else (ny, nx, qy)
    T = 8 if L > 1024 else 16
    return Q >= 16 and P * ((Q + T - 1) // T) > TURNS[L] * CTAS_PER_SM[L] * sms


@pytest.mark.parametrize("shape,basis,axes", CASES)
def test_every_variant_matches_the_oracle(oracle_mod, shape, basis, axes):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1805_07801_gb300 import build as b

    b.build()
    import paper_1805_07801_gb300 as fk

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert all(takes_the_pipeline(shape, basis, a, sms) for a in axes)
    nx, ny, nz = shape
    half = basis[2] == "F"
    f = synth.uniform_pm1(64, 0, shape)
    plan = fk.fftk_plan_create(nx, ny, nz)
    try:
        x = torch.from_numpy(np.ascontiguousarray(f, dtype=np.float32)).to("cuda:0")
        F = torch.empty((nx, ny, nz // 2 + 1, 2) if half else shape, dtype=torch.float32, device="cuda:0")
        y = torch.empty_like(x)
        for _ in range(2):
            F.zero_()
            y.zero_()
            fk.fftk_forward(plan, basis, x.data_ptr(), F.data_ptr(), 1, stream())
            fk.fftk_inverse(plan, basis, F.data_ptr(), y.data_ptr(), 1, stream())
        fk.fftk_sync(plan, stream())
        sync()
        Fg = from_dev_c64(F) if half else F.cpu().numpy().astype(np.float64)
        yg = y.cpu().numpy()
    finally:
        fk.fftk_plan_destroy(plan)
    want = oracle_mod.rfft3(f.astype(np.float64)) if basis == "FFF" else oracle_mod.transform3(f.astype(np.float64), basis)
    assert rel_l2(Fg, want) < 2e-6
    assert np.max(np.abs(Fg - want)) < 1e-5 * np.max(np.abs(want))
    assert rel_l2(yg, f) < 2e-6
    assert np.max(np.abs(yg - f)) < 1e-5
