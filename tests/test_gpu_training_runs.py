"""The training gradient of batches far beyond one wave of CTAs: its FP32 sums
take 64 samples and then at most 14 chunk totals, and everything longer is added
in FP64.  With equal samples and a power-of-two batch every chunk's total is the
one-chunk gradient divided by a power of two, so the exact sum is known: 14 equal
terms added one after the other are off by less than (2 + ... + 14) / 14 < 7.5
units of 2^-24, the rounding of the result adds one.
"""
import numpy as np
import pytest

from gpu_helpers import stream, sync

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log2_batch", [15, 18, 19, 21])
def test_long_batches_add_in_fp64(log2_batch):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1805_07801_gb300 import build as b

    b.build()
    import paper_1805_07801_gb300 as fk

    rng = np.random.default_rng(7)
    p = np.concatenate([rng.uniform(-1, 1, n) / np.sqrt(d) for n, d in ((384, 5), (4160, 64), (4160, 64), (390, 64))])
    pd = torch.from_numpy(p.astype(np.float32)).to("cuda:0")
    x1 = torch.from_numpy(rng.standard_normal(5).astype(np.float32)).to("cuda:0")
    t1 = torch.from_numpy(rng.standard_normal(6).astype(np.float32)).to("cuda:0")
    B = 1 << log2_batch
    x, t = x1.repeat(B, 1).contiguous(), t1.repeat(B, 1).contiguous()
    one, all_ = torch.zeros(9094, device="cuda:0"), torch.zeros(9094, device="cuda:0")
    loss = torch.zeros(2, dtype=torch.float64, device="cuda:0")
    ctx = fk.tarang_mlp_create(B)
    try:
        fk.tarang_mlp_loss_grad(ctx, pd.data_ptr(), x.data_ptr(), t.data_ptr(), 64, one.data_ptr(), loss.data_ptr(),
                                stream())
        fk.tarang_mlp_loss_grad(ctx, pd.data_ptr(), x.data_ptr(), t.data_ptr(), B, all_.data_ptr(),
                                loss.data_ptr() + 8, stream())
        sync()
    finally:
        fk.tarang_mlp_destroy(ctx)
    g1, gB = one.cpu().numpy().astype(np.float64), all_.cpu().numpy().astype(np.float64)
    assert np.count_nonzero(g1) > 9000
    assert np.all(np.abs(gB - g1) <= 8.5 * 2.0 ** -24 * np.abs(g1))
    l1, lB = loss.cpu().numpy()
    assert abs(lB - l1) <= 1e-13 * l1
