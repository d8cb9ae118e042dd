"""Workspaces between the smallest accepted and the full one: intervals in the least space a
layer at a time, chunks of several layers, leaves alone; the same sums and adjoints as on the
full workspace up to the order of the terms (1e-12 in FP64, 2e-6 in FP32)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda")


@pytest.mark.parametrize("n,N", [(2048, 33), (2047, 700), (2048, 2049), (9000, 3000)])
@pytest.mark.parametrize("prec", [0, 1])
def test_every_workspace_gives_the_same(n, N, prec):
    from paper_2105_14782_gb300 import xs
    L = 5
    dl = xs.DeviceLines(W.water_like(n, seed=n))
    nu, P = dev(W.grid_lognu(N)), dev(10.0 ** np.linspace(-3, 2, L))
    T = dev(np.linspace(700.0, 1900.0, L))
    full, least = xs.workspace_bytes(n, N, L, prec), xs.lib().xs_workspace_min_bytes(n, N, L, prec)
    lam = dev(1e20 * (1.0 + 0.5 * np.random.default_rng(7).uniform(size=(L, N))))
    want = xs.xs_compute(dl, nu, T, P, 1.1, 3.0, prec).double()
    g_T, g_b = xs.xs_compute_adjoint(dl, nu, T, P, lam, 1.1, 3.0, prec)
    tol = 2e-6 if prec else 1e-12
    for size in (least, least - 256, (least + full) // 2, full - 256):
        ws = torch.empty(size, dtype=torch.uint8, device="cuda")
        try:
            got = xs.xs_compute(dl, nu, T, P, 1.1, 3.0, prec, workspace=ws).double()
        except xs.XsError as e:  # below the smallest list's only plan
            assert e.code == xs.XS_EINVAL and n < 2048 and size == least - 256
            continue
        assert torch.all((got - want).abs() <= tol * want)
        a, b = xs.xs_compute_adjoint(dl, nu, T, P, lam, 1.1, 3.0, prec, workspace=ws)
        big = max(float((g_T * T).abs().max()), abs(g_b.item()))
        assert float(((a - g_T) * T).abs().max()) <= tol * big and abs((b - g_b).item()) <= tol * big
