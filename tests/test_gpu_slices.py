"""Few leaves with long lists, whose near lines several blocks share: grids of a few points,
coarse ones on which no line covers a leaf and fine ones, one layer and several, and models
that mix such a list with a short one; against the oracle."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda")


@pytest.mark.parametrize("N,span,cut", [(1, 0.0, 1.0), (33, 200.0, 5.0), (64, 0.3, 25.0), (130, 40.0, 2.0)])
@pytest.mark.parametrize("n,L", [(16384, 1), (30001, 3)])
def test_long_lists_on_few_points(n, L, N, span, cut):
    from paper_2105_14782_gb300 import xs
    nu = np.linspace(4400.0, 4400.0 + span, N)
    lines = W.water_like(n, seed=n + N, nu_min=4400.0 - cut, nu_max=4400.0 + span + cut)
    P, T = np.array([1.0, 1e-3, 30.0])[:L], np.array([1200.0, 700.0, 1900.0])[:L]
    want = oracle.xs(lines, nu, T, P, sb=1.3, wing_cut=cut)
    m = want > 1e-6 * want.max(axis=1, keepdims=True)
    dl = xs.DeviceLines(lines)
    args = dl, dev(nu), dev(T), dev(P)
    lam = dev(1e20 * (1.0 + 0.5 * np.random.default_rng(7).uniform(size=(L, N))))
    grad = {}
    for prec, tol in ((xs.PREC_FP64, 1e-10), (xs.PREC_MIXED, 1e-5)):
        got = xs.xs_compute(*args, 1.3, cut, prec).double().cpu().numpy()
        assert np.max(np.abs(got - want)[m] / want[m]) < tol
        small = torch.empty(xs.lib().xs_workspace_min_bytes(n, N, L, prec), dtype=torch.uint8, device="cuda")
        for name, ws in (("full", None), ("small", small)):
            g_T, g_b = xs.xs_compute_adjoint(*args, lam, 1.3, cut, prec, workspace=ws)
            grad[prec, name] = np.append(g_T.cpu().numpy() * T, g_b.cpu().numpy())
    ref = grad[xs.PREC_FP64, "small"]
    big = np.max(np.abs(ref))
    assert np.max(np.abs(grad[xs.PREC_FP64, "full"] - ref)) <= 1e-10 * big
    for name in ("full", "small"):
        assert np.max(np.abs(grad[xs.PREC_MIXED, name] - ref)) <= 1e-4 * big


@pytest.mark.parametrize("sizes", [(20000, 300), (300, 20000, 18000)])
def test_models_that_mix_them_with_short_lists(sizes):
    from paper_2105_14782_gb300 import xs
    L, N = 4, 70
    p, dp = W.pressure_layers(L)
    nu = W.grid_lognu(N, 4363.0, 4367.0)
    species = [W.water_like(n, seed=60 + k, nu_min=4361.0, nu_max=4369.0) for k, n in enumerate(sizes)]
    atm = W.Atmosphere(species=species, vmr=[1e-3] * len(sizes), nu=nu, p_bar=p, dp_bar=dp, wing_cut=2.0)
    theta = np.array([1250.0, 0.12] + [-2.8 - 0.2 * k for k in range(len(sizes))] + [1.3])
    F0 = oracle.forward(atm, theta)
    sig = 0.01 * F0
    d = F0 + sig * W.std_normal(N)
    ll_o, g_o, F_o = oracle.logl_grad(atm, theta, d, sig)
    for prec, tol_f, tol_g in ((xs.PREC_FP64, 1e-10, 1e-8), (xs.PREC_MIXED, 1e-6, 1e-4)):
        model = xs.EmissionModel(atm, prec=prec, d_obs=d, sig_obs=sig)
        F = model.forward(theta).cpu().numpy()
        assert np.max(np.abs(F - F_o) / F_o) < tol_f
        _, g = model.logl_grad(theta)
        assert np.all(np.abs(g - g_o) <= tol_g * np.abs(g_o) + 1e-12 * np.abs(g_o).max()), (prec, g, g_o)
