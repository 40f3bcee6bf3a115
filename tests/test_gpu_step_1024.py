"""One step at 1024^3 (every update mode of the forward x passes at that size)
against the same step at 256^3, for states with |k_i| <= 5: a right-hand side at
most doubles the band, so even RK4's last stage has |k_i| <= 80, inside the 2/3
set of both grids (85 and 341) with aliases outside it, and both grids hold the
same Fourier coefficients.  The 256^3 step is held to the oracle by other tests.
Tolerance: a right-hand side within 1e-5 of the exact one on each grid, times
dt |N| / |u| <= 0.1: relative L2 2e-6 of the state; the modes that only the
large grid holds stay below 1e-6 of the largest coefficient.
"""
import pytest

from gpu_helpers import stream, sync

pytestmark = pytest.mark.gpu

BAND, DT = 5, 0.02


def _state(n, fields):
    """The same random band-limited spectrum on every grid."""
    import torch

    g = torch.Generator().manual_seed(3)
    m = 16
    k = torch.fft.fftfreq(m, 1.0 / m)
    keep = (k.abs() <= BAND)[:, None, None] & (k.abs() <= BAND)[None, :, None] & (torch.arange(m // 2 + 1) <= BAND)
    small = torch.fft.rfftn(torch.randn((fields, m, m, m), generator=g, dtype=torch.float64), dim=(1, 2, 3),
                            norm="forward") * keep
    kx, ky, kz = k[:, None, None].double(), k[None, :, None].double(), torch.arange(m // 2 + 1).double()[None, None, :]
    k2 = kx * kx + ky * ky + kz * kz
    k2[0, 0, 0] = 1.0
    d = (kx * small[0] + ky * small[1] + kz * small[2]) / k2
    for f, w in enumerate((kx, ky, kz)):
        small[f] -= w * d
    small[:, 0, 0, 0] = 0
    u = torch.zeros((fields, n, n, n // 2 + 1), dtype=torch.complex64, device="cuda:0")
    idx = k.long() % n
    u[:, idx[:, None, None], idx[None, :, None], torch.arange(m // 2 + 1)[None, None, :]] = small.to(
        torch.complex64).to("cuda:0")
    return u


def _step(fk, n, kind, scheme):
    plan = fk.fftk_plan_create(n, n, n)
    try:
        u = _state(n, 4 if kind == "rbc" else 3)
        if kind == "rbc":
            fk.tarang_rbc_step(plan, u.data_ptr(), 1e4, 1.0, DT, 1, scheme, stream(), fk.TARANG_RBC_FFF)
        else:
            fk.tarang_ns_step(plan, u.data_ptr(), fk.make_params(1e-2, DT, scheme=scheme), 1, False, stream())
        sync()
    finally:
        fk.fftk_plan_destroy(plan)
    return u


@pytest.mark.parametrize("kind", ["ns", "rbc"])
@pytest.mark.parametrize("scheme", ["rk2", "rk4"])
def test_step_of_a_band_limited_state(kind, scheme):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1805_07801_gb300 import build as b

    b.build()
    import paper_1805_07801_gb300 as fk

    s = fk.TARANG_RK2 if scheme == "rk2" else fk.TARANG_RK4
    small, large = _step(fk, 256, kind, s), _step(fk, 1024, kind, s)
    moved = (small - _state(256, small.shape[0])).abs().square().sum().sqrt() / small.abs().square().sum().sqrt()
    assert 1e-3 < float(moved) < 0.1
    idx = torch.fft.fftfreq(256, 1.0 / 256).long().to("cuda:0")
    same = (torch.arange(256, device="cuda:0") != 128).nonzero()[:, 0]  # the Nyquist rows have no counterpart
    kz = torch.arange(128, device="cuda:0")
    top = float(small.abs().max())
    for f in range(small.shape[0]):
        a = small[f][same][:, same][:, :, kz]
        rows = idx[same] % 1024
        c = large[f][rows][:, rows][:, :, kz]
        err = float((a - c).abs().square().sum().sqrt() / a.abs().square().sum().sqrt())
        assert err < 2e-6, (f, err)
        large[f][rows[:, None, None], rows[None, :, None], kz[None, None, :]] = 0
        assert float(large[f].abs().max()) < 1e-6 * top
