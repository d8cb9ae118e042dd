"""MODIT with transforms shorter and a little longer than a block's frequencies (64 threads of
8 and of 4), one and several layers, forward against the oracle and adjoint against the
forward's differences; with the tolerances of the other MODIT tests."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda")


@pytest.mark.parametrize("N,n_fft", [(20, 64), (100, 256), (200, 512), (400, 1024), (900, 2048)])
@pytest.mark.parametrize("L,ng", [(1, 1), (3, 5)])
def test_short_transforms(N, n_fft, L, ng):
    from paper_2105_14782_gb300 import xs
    lo, hi = 4364.0, 4364.0 + 0.002 * N
    lines = W.water_like(60, seed=N, nu_min=lo, nu_max=hi)
    P, T = np.array([1.0, 0.01, 10.0])[:L], np.array([1200.0, 800.0, 1700.0])[:L]
    dl = xs.DeviceLines(lines)
    want = oracle.modit(lines, lo, hi, N, T, P, n_gamma=ng, n_fft=n_fft)
    got = xs.modit_compute(dl, lo, hi, N, dev(T), dev(P), n_gamma=ng, n_fft=n_fft).cpu().numpy()
    assert np.max(np.abs(got - want)) < 1e-10 * np.max(np.abs(want))
    lam = dev((1.0 + 0.5 * np.random.default_rng(N).uniform(size=(L, N))) / want.max())
    _, g_b = xs.modit_compute_adjoint(dl, lo, hi, N, dev(T), dev(P), lam, n_gamma=ng, n_fft=n_fft)
    up, dn = (float((lam * xs.modit_compute(dl, lo, hi, N, dev(T), dev(P), broad_scale=1.0 + s, n_gamma=ng,
                                            n_fft=n_fft)).sum()) for s in (1e-4, -1e-4))
    assert g_b.item() == pytest.approx((up - dn) / 2e-4, rel=1e-5, abs=1e-7 * L * N)
