"""Lists without far sets: below and above the lengths from which intervals are used (256
lines, 64 in FP64) and from which a leaf's window is split (96 lines), full and partial
windows, lines on both sides of a leaf's cut edges; against the oracle, adjoints against
FP64 with the intervals off and on."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

P = np.array([1e-3, 0.3, 30.0])
T = np.array([700.0, 1200.0, 1900.0])


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda")


@pytest.mark.parametrize("n", [1, 33, 63, 64, 95, 96, 97, 200, 255])
@pytest.mark.parametrize("N,cut", [(33, 25.0), (700, 25.0), (700, 3.0), (1500, 0.5)])
def test_short_lists(n, N, cut):
    from paper_2105_14782_gb300 import xs
    nu = W.grid_lognu(N, 4360.0, 4370.0)
    lines = W.water_like(n, seed=n, nu_min=4355.0, nu_max=4375.0)
    want = oracle.xs(lines, nu, T, P, sb=1.3, wing_cut=cut)
    m = want > 1e-6 * want.max(axis=1, keepdims=True)
    dl = xs.DeviceLines(lines)
    args = dl, dev(nu), dev(T), dev(P)
    lam = dev(1e20 * (1.0 + 0.5 * np.random.default_rng(7).uniform(size=(3, N))))
    grad = {}
    for prec, tol in ((xs.PREC_FP64, 1e-10), (xs.PREC_MIXED, 1e-5)):
        got = xs.xs_compute(*args, 1.3, cut, prec).double().cpu().numpy()
        assert np.all((got == 0) == (want == 0))
        assert m.sum() == 0 or np.max(np.abs(got - want)[m] / want[m]) < tol
        small = torch.empty(xs.lib().xs_workspace_min_bytes(n, N, 3, prec), dtype=torch.uint8, device="cuda")
        for name, ws in (("full", None), ("small", small)):
            g_T, g_b = xs.xs_compute_adjoint(*args, lam, 1.3, cut, prec, workspace=ws)
            grad[prec, name] = np.append(g_T.cpu().numpy() * T, g_b.cpu().numpy())
    ref = grad[xs.PREC_FP64, "small"]
    big = np.max(np.abs(ref))
    assert np.max(np.abs(grad[xs.PREC_FP64, "full"] - ref)) <= 1e-10 * big
    for name in ("full", "small"):
        assert np.max(np.abs(grad[xs.PREC_MIXED, name] - ref)) <= 1e-4 * big
