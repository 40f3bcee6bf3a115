"""The fused solver passes at 384^3 (lines of 24 values per thread, y passes
pipelined through the mixed-radix engine): right-hand sides of Navier-Stokes and
of periodic convection for band-limited states.  With |k_i| <= 21 the products
reach |k_i| <= 42 and are alias-free and kept on a 128^3 grid as on a 384^3 one,
so the oracle's 128^3 result fixes every 384^3 coefficient.  Relative L2 1e-5, as
for every right-hand side.
"""
import numpy as np
import pytest

import synth
from gpu_helpers import empty_c64, from_dev_c64, rel_l2, stream, to_dev_c64

pytestmark = pytest.mark.gpu


def _embed(u, N):
    n = u.shape[1]
    a = np.arange(n)
    a = a[2 * a != n]
    big = np.where(2 * a < n, a, a - n + N)
    out = np.zeros((u.shape[0], N, N, N // 2 + 1), dtype=u.dtype)
    for c in range(u.shape[0]):
        out[c][np.ix_(big, big, np.arange(n // 2 + 1))] = u[c][np.ix_(a, a, np.arange(n // 2 + 1))]
    return out


def _inside(big, n):
    N = big.shape[1]
    a = np.arange(n)
    a = a[2 * a != n]
    rows = np.where(2 * a < n, a, a - n + N)
    sub = np.zeros((big.shape[0], n, n, n // 2 + 1), dtype=big.dtype)
    for c in range(big.shape[0]):
        sub[c][np.ix_(a, a, np.arange(n // 2 + 1))] = big[c][np.ix_(rows, rows, np.arange(n // 2 + 1))]
    return sub


@pytest.mark.parametrize("kind", ["ns", "rbc"])
def test_rhs_384_band_limited_matches_oracle_at_128(oracle_mod, kind):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1805_07801_gb300 import build as b

    b.build()
    import paper_1805_07801_gb300 as fk

    n, N = 64, 384
    u = oracle_mod.ic_random(synth.normal_fields(17, 3, (n, n, n)), k0=8.0, E0=0.5).astype(np.complex64)
    if kind == "rbc":
        th = oracle_mod.ic_random(synth.normal_fields(18, 3, (n, n, n)), k0=8.0, E0=0.5).astype(np.complex64)
        u = np.concatenate([u, th[:1]])
    want = (oracle_mod.ns_rhs if kind == "ns" else oracle_mod.rbc_rhs)(_embed(u, 128).astype(np.complex128))
    plan = fk.fftk_plan_create(N, N, N)
    try:
        ud = to_dev_c64(_embed(u, N))
        out = empty_c64((u.shape[0], N, N, N // 2 + 1))
        if kind == "ns":
            fk.tarang_ns_rhs(plan, ud.data_ptr(), out.data_ptr(), fk.make_params(0.0), stream())
        else:
            fk.tarang_rbc_rhs(plan, ud.data_ptr(), out.data_ptr(), stream())
        fk.fftk_sync(plan, stream())
        got = from_dev_c64(out)
    finally:
        fk.fftk_plan_destroy(plan)
    sub = _inside(got, 128)
    assert rel_l2(sub, want) < 1e-5
    total = np.sqrt(sum(float(np.sum(np.abs(g.astype(np.complex128)) ** 2)) for g in got))
    rest = np.sqrt(max(0.0, total ** 2 - float(np.linalg.norm(sub.ravel().astype(np.complex128))) ** 2))
    assert rest < 1e-5 * np.linalg.norm(want.ravel())
