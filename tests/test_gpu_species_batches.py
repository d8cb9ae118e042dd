"""Models whose species run their line sums together or apart: empty lists, lists below and
above the length from which far lines go to nodes, and dense and sparse lists (intervals
halved or quartered) side by side; against the FP64 oracle, with the tolerances of the
composite model's other cases."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("sizes", [(0, 300), (300, 0, 700), (100, 300, 90), (5000, 260, 0, 4800)])
def test_mixed_lists_match_the_oracle(sizes):
    from paper_2105_14782_gb300 import xs
    L, N = 4, 600
    p, dp = W.pressure_layers(L)
    nu = W.grid_lognu(N, 4363.0, 4367.0)
    species = [W.water_like(n, seed=60 + k, nu_min=4361.0, nu_max=4369.0) for k, n in enumerate(sizes)]
    atm = W.Atmosphere(species=species, vmr=[1e-3] * len(sizes), nu=nu, p_bar=p, dp_bar=dp, wing_cut=2.0)
    theta = np.array([1250.0, 0.12] + [-2.8 - 0.2 * k for k in range(len(sizes))] + [1.3])
    F0 = oracle.forward(atm, theta)
    sig = 0.01 * F0
    d = F0 + sig * W.std_normal(N)
    ll_o, g_o, F_o = oracle.logl_grad(atm, theta, d, sig)
    scale = np.abs(g_o)
    for prec, tol_f, tol_g in ((xs.PREC_FP64, 1e-10, 1e-8), (xs.PREC_MIXED, 1e-6, 1e-4)):
        model = xs.EmissionModel(atm, prec=prec, d_obs=d, sig_obs=sig)
        F = model.forward(theta).cpu().numpy()
        assert np.max(np.abs(F - F_o) / F_o) < tol_f
        ll, g = model.logl_grad(theta)
        assert ll == pytest.approx(oracle.loglike(F, d, sig), rel=1e-12)
        assert np.all(np.abs(g - g_o) <= tol_g * scale + 1e-12 * scale.max()), (prec, g, g_o)
