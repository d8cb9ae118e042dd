"""The composite model's MODIT adjoint takes the forward's distribution: the same bits as
when the sweep is repeated, and the gradients of the standalone calls, which form it
themselves (the same kernels on the same inputs); for one and several gamma' nodes."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec,n_gamma,N", [(0, 1, 1500), (0, 16, 1501), (1, 5, 2047)])
def test_vjp_repeats_and_matches_the_standalone_adjoint(prec, n_gamma, N):
    from paper_2105_14782_gb300 import xs
    lo, hi = 4364.0, 4366.0
    p, dp = W.pressure_layers(12)
    nu = W.grid_lognu(N, lo, hi)
    atm = W.Atmosphere(species=[W.water_like(400, seed=5, nu_min=4363.5, nu_max=4366.5)], vmr=[1e-3], nu=nu, p_bar=p,
                       dp_bar=dp)
    theta = [1300.0, 0.1, -3.0, 1.2]
    m = xs.EmissionModel(atm, prec=prec, method="modit", n_gamma=n_gamma)
    F = m.forward_keep(theta).clone()
    g = torch.as_tensor(np.random.default_rng(1).standard_normal(N), device="cuda")
    a = m.vjp(theta, g).clone()
    b = m.vjp(theta, g).clone()
    assert torch.equal(a, b)
    assert torch.equal(F, m.forward(theta))
    # the same chain from the standalone calls
    dl = m.species[0]
    T = xs.layer_temperatures(theta[0], theta[1], m.P)
    n_fft = xs.modit_fft_length(lo, hi, N, dl)
    sig = xs.modit_compute(dl, float(nu[0]), float(nu[-1]), N, T, m.P, theta[3], n_gamma, n_fft, prec)
    vmr = torch.full((1, 12), 10.0 ** theta[2], dtype=torch.float64, device="cuda")
    dtau = xs.tau_layers([sig], vmr, m.P, m.dP, prec=prec)
    g_dtau, _ = xs.emission_spectrum_adjoint(g, dtau, T, m.nu)
    gs, gv = xs.tau_layers_adjoint([sig], vmr, m.P, m.dP, g_dtau, prec=prec)
    _, g_b = xs.modit_compute_adjoint(dl, float(nu[0]), float(nu[-1]), N, T, m.P, gs[0], theta[3], n_gamma, n_fft, prec)
    assert a[3].item() == pytest.approx(g_b.item(), rel=1e-12)
    assert a[2].item() == pytest.approx(float(np.log(10.0) * (gv[0] * vmr[0]).sum().item()), rel=1e-12)
