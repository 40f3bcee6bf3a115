"""The training kernel's chunks of 64 samples: batches below, at and above one
chunk, one beyond the persistent grid (304 chunks) and a ragged one that takes
several rounds, against the FP64 oracle.  FP32 test mode (layer inputs not
rounded): every gradient tensor within 1e-5, as for the other training tests.
"""
import numpy as np
import pytest

from gpu_helpers import rel_l2, stream, sync

pytestmark = pytest.mark.gpu

TENSORS = {"W1": (0, 320), "b1": (320, 384), "W2": (384, 4480), "b2": (4480, 4544), "W3": (4544, 8640),
           "b3": (8640, 8704), "W4": (8704, 9088), "b4": (9088, 9094)}


@pytest.mark.parametrize("B", [1, 63, 64, 65, 304 * 64 + 1, 2 * 304 * 64 + 777])
def test_gradient_and_step_of_every_batch_size(oracle_mod, B):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1805_07801_gb300 import build as b

    b.build()
    import paper_1805_07801_gb300 as fk

    rng = np.random.default_rng(B)
    p = np.concatenate([rng.uniform(-1, 1, n) / np.sqrt(d) for n, d in ((384, 5), (4160, 64), (4160, 64), (390, 64))])
    p = p.astype(np.float32)
    x = rng.standard_normal((B, 5)).astype(np.float32)
    t = rng.standard_normal((B, 6)).astype(np.float32)
    # offset by one float: the data may start on any 4-byte boundary
    xd = torch.zeros(5 * B + 1, device="cuda:0")[1:].copy_(torch.from_numpy(x).reshape(-1))
    td = torch.zeros(6 * B + 1, device="cuda:0")[1:].copy_(torch.from_numpy(t).reshape(-1))
    pd = torch.from_numpy(p).to("cuda:0")
    g, loss = torch.zeros(9094, device="cuda:0"), torch.zeros(1, dtype=torch.float64, device="cuda:0")
    ctx = fk.tarang_mlp_create(B)
    try:
        fk.tarang_mlp_loss_grad_mode(ctx, pd.data_ptr(), xd.data_ptr(), td.data_ptr(), B, g.data_ptr(),
                                     loss.data_ptr(), fk.TARANG_ACT_FP32, stream())
        # one training step against the gradient (BF16 inputs) and Adam as calls of their own
        gb = torch.zeros_like(g)
        fk.tarang_mlp_loss_grad(ctx, pd.data_ptr(), xd.data_ptr(), td.data_ptr(), B, gb.data_ptr(), 0, stream())
        pa, ma, va = pd.clone(), torch.zeros_like(g), torch.zeros_like(g)
        pb, mb, vb = pd.clone(), torch.zeros_like(g), torch.zeros_like(g)
        fk.tarang_mlp_adam(pa.data_ptr(), ma.data_ptr(), va.data_ptr(), gb.data_ptr(), 1, 1e-3, 0.9, 0.999, 1e-8,
                           stream())
        fk.tarang_mlp_train_step(ctx, pb.data_ptr(), mb.data_ptr(), vb.data_ptr(), 1, xd.data_ptr(), td.data_ptr(), B,
                                 1e-3, 0, stream())
        sync()
    finally:
        fk.tarang_mlp_destroy(ctx)
    lo, go = oracle_mod.mlp_loss_grad(p.astype(np.float64), x.astype(np.float64), t.astype(np.float64),
                                      bf16_acts=False)
    assert abs(float(loss) - lo) < 1e-6 * lo
    gg = g.cpu().numpy().astype(np.float64)
    for name, (i, j) in TENSORS.items():
        assert rel_l2(gg[i:j], go[i:j]) < 1e-5, name
    assert torch.equal(pa, pb) and torch.equal(ma, mb) and torch.equal(va, vb)
