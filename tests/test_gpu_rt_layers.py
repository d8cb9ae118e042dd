"""Emission and its adjoint where the kernels change the points of a block with the number
of layers (segments without layers, one layer in some of a warp's segments), against the
oracle; the adjoint against its parts."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda")


@pytest.mark.parametrize("L,N", [(1, 4096), (3, 9001), (8, 2000), (15, 2003), (16, 2003), (20, 2003), (24, 5001), (33, 7)])
def test_emission_with_few_layers(L, N):
    from paper_2105_14782_gb300 import xs
    rng = np.random.default_rng(L)
    dtau, T, nu = rng.lognormal(-1.0, 2.0, (L, N)), rng.uniform(500.0, 2000.0, L), W.grid_lognu(N)
    F = xs.emission_spectrum(dev(dtau), dev(T), dev(nu)).cpu().numpy()
    want = oracle.emission(dtau, T, nu)
    assert np.max(np.abs(F - want) / want) < 1e-13
    # the adjoint of single points equals that of the whole grid (other blocks), and its sums
    # over the points those of two halves (1e-12 of the largest)
    lam = np.abs(rng.standard_normal(N))
    gd, gT = xs.emission_spectrum_adjoint(dev(lam), dev(dtau), dev(T), dev(nu))
    cut = max(1, N // 3)
    parts = [xs.emission_spectrum_adjoint(dev(lam[q]), dev(dtau[:, q]), dev(T), dev(nu[q]))
             for q in (slice(0, cut), slice(cut, N))]
    joined = torch.cat([q[0] for q in parts], dim=1)
    assert torch.all((gd - joined).abs() <= 1e-12 * joined.abs().amax(dim=0, keepdim=True))
    assert torch.allclose(gT, parts[0][1] + parts[1][1], rtol=1e-12, atol=1e-12 * float(gT.abs().max()))
