"""Responses onto grids whose points lie much further apart than a kernel's support, where
each point reads its own support instead of the block's tiles; with the tolerances of the
blocked kernels' test."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def dev(a):
    return torch.as_tensor(np.array(a, dtype=np.float64, order="C", copy=True), device="cuda")


def grid(N, width):
    return 4360.0 * (1.0 + width / 4360.0) ** (np.arange(N) / (N - 1))


@pytest.mark.parametrize("N,n_out,beta", [(40000, 20, 2.6), (40000, 200, 0.7), (5000, 17, 1.0)])
def test_ip_rv_against_the_oracle(N, n_out, beta):
    from paper_2105_14782_gb300 import xs
    rng = np.random.default_rng(n_out)
    nu = grid(N, 100.0)
    out = np.sort(rng.uniform(4361.0, 4459.0, n_out))
    F = 1.0 + 0.4 * np.sin(7.0 * (nu - nu[0])) * np.cos(0.9 * nu)
    want = oracle.ip_rv(F, nu, out, beta, 3.0)
    got = xs.response_ip_rv(dev(F), dev(nu), dev(out), beta, 3.0).cpu().numpy()
    assert np.max(np.abs(got / want - 1)) < 1e-11
    g = rng.standard_normal(n_out)
    gF, g_rv = xs.response_ip_rv_adjoint(dev(g), dev(F), dev(nu), dev(out), beta, 3.0)
    assert abs(gF.cpu().numpy() @ F - g @ want) <= 1e-11 * np.abs(g) @ want
    h = 1e-4 * beta
    up, lo = (oracle.ip_rv(F, nu, out, beta, 3.0 + s * h) for s in (1.0, -1.0))
    assert g_rv.item() == pytest.approx(g @ (up - lo) / (2 * h), rel=1e-5, abs=1e-6 * np.abs(g).sum() / beta)


def test_many_points_against_few_at_a_time():
    """8,192 points and more take four lanes a point, fewer 16: the same points in parts."""
    from paper_2105_14782_gb300 import xs
    N, n_out = 400000, 8300
    nu, rng = grid(N, 1000.0), np.random.default_rng(1)
    out = np.sort(rng.uniform(4370.0, 5350.0, n_out))
    F = 1.0 + 0.4 * np.sin(7.0 * (nu - nu[0])) * np.cos(0.9 * nu)
    got = xs.response_ip_rv(dev(F), dev(nu), dev(out), 0.3, 3.0)
    parts = torch.cat([xs.response_ip_rv(dev(F), dev(nu), dev(out[q]), 0.3, 3.0)
                       for q in (slice(0, 4000), slice(4000, n_out))])
    assert float((got / parts - 1).abs().max()) < 1e-13
