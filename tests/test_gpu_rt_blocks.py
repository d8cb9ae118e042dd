"""Transfer on both sides of the grid sizes at which the emission kernels change the points
of a block (608 blocks of 16 and of 32 points), on grids that end inside a block; the sums
over the grid (adjoint of the optical depth, likelihood) there as well."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda")


@pytest.mark.parametrize("N", [7, 608 * 16 - 1, 608 * 16, 608 * 32 - 1, 608 * 32 + 1])
def test_transfer_at_the_block_sizes(N):
    from paper_2105_14782_gb300 import xs
    L = 5
    rng = np.random.default_rng(N)
    s = rng.lognormal(-48.0, 3.0, (2, L, N))
    P, dP = W.pressure_layers(L)
    vmr = np.array([[1e-3] * L, [5e-4] * L])
    dtau = oracle.tau(list(s), vmr, P, dP)
    got = xs.tau_layers([dev(s[0]), dev(s[1])], dev(vmr), dev(P), dev(dP), prec=xs.PREC_FP64)
    assert np.allclose(got.cpu().numpy(), dtau, rtol=1e-14, atol=0)
    T, nu = np.linspace(700.0, 1900.0, L), W.grid_lognu(N)
    F = xs.emission_spectrum(dev(dtau), dev(T), dev(nu))
    want = oracle.emission(dtau, T, nu)
    assert np.max(np.abs(F.cpu().numpy() - want) / want) < 1e-13
    # adjoint: points are independent, so columns equal those of a short grid's blocks up
    # to rounding, and the sums over points those of two halves (1e-12 of the terms' sum)
    lam = np.abs(rng.standard_normal(N))
    gd, gT = xs.emission_spectrum_adjoint(dev(lam), dev(dtau), dev(T), dev(nu))
    cut = max(1, N // 3)
    parts = [xs.emission_spectrum_adjoint(dev(lam[q]), dev(dtau[:, q]), dev(T), dev(nu[q]))
             for q in (slice(0, cut), slice(cut, N))]
    joined = torch.cat([q[0] for q in parts], dim=1)
    assert torch.all((gd - joined).abs() <= 1e-12 * joined.abs().amax(dim=0, keepdim=True))
    assert torch.allclose(gT, parts[0][1] + parts[1][1], rtol=1e-12, atol=1e-12 * float(gT.abs().max()))
    gs, gv = xs.tau_layers_adjoint([dev(s[0]), dev(s[1])], dev(vmr), dev(P), dev(dP), gd, prec=xs.PREC_FP64)
    chain = s * gs[0].cpu().numpy()[None] / vmr[0][None, :, None]
    terms = chain.sum(axis=2), np.abs(chain).sum(axis=2)
    assert np.all(np.abs(gv.cpu().numpy() - terms[0]) <= 1e-12 * terms[1])
    d, e = want * (1 + 0.01 * rng.standard_normal(N)), 0.01 * want
    ll, gF = xs.loglike_gauss(F, dev(d), dev(e))
    Fn = F.cpu().numpy()
    assert ll.item() == pytest.approx(oracle.loglike(Fn, d, e), rel=1e-13)
    assert np.allclose(gF.cpu().numpy(), (d - Fn) / e ** 2, rtol=1e-14)


@pytest.mark.parametrize("L", [1, 5, 40])
def test_bottom_layer_on_its_own_temperature(L):
    """The bottom source has the last layer's temperature, so F0 does not depend on that
    layer's optical depth: its derivative is a difference of equal terms, exactly zero."""
    from paper_2105_14782_gb300 import xs
    N = 1003
    rng = np.random.default_rng(L)
    dtau, lam = rng.lognormal(-1.0, 2.0, (L, N)), rng.standard_normal(N)
    gd, _ = xs.emission_spectrum_adjoint(dev(lam), dev(dtau), dev(rng.uniform(400.0, 2000.0, L)), dev(W.grid_lognu(N)))
    assert torch.all(gd[L - 1] == 0.0)
