"""Responses where the blocked kernels can go wrong: one output point, counts around a
block's 8 and 32 points, output points outside the grid's support, an unsorted output
grid, supports longer than a staged tile, and grids so coarse that a block spans many
supports."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def xs():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2105_14782_gb300 import xs as m
    return m


def dev(a):
    return torch.as_tensor(np.array(a, dtype=np.float64, order="C", copy=True), device="cuda")


def spectrum(nu):
    return 1.0 + 0.4 * np.sin(7.0 * (nu - nu[0])) * np.cos(0.9 * nu)


@pytest.mark.parametrize("N,n_out,beta,width", [(4000, 1, 2.6, 10.0), (4000, 7, 2.6, 10.0), (4000, 33, 2.6, 10.0),
                                                (20000, 9, 25.0, 10.0), (9000, 8193, 0.9, 10.0), (300, 257, 900.0, 2000.0)])
def test_ip_rv_against_the_oracle(xs, N, n_out, beta, width):
    """1e-11: a pair's velocity is accurate to 1e-16 c (the ratio's rounding, 3e-11 km/s), at most
    4e-11 of beta here, and enters through contrasts below one."""
    rng = np.random.default_rng(N + n_out)
    nu = 4360.0 * (1.0 + width / 4360.0) ** (np.arange(N) / (N - 1))
    out = np.sort(rng.uniform(nu[0] + 0.2 * width, nu[-1] - 0.2 * width, n_out))
    F = spectrum(nu)
    want = oracle.ip_rv(F, nu, out, beta, 3.0)
    got = xs.response_ip_rv(dev(F), dev(nu), dev(out), beta, 3.0).cpu().numpy()
    assert np.max(np.abs(got / want - 1)) < 1e-11
    back = xs.response_ip_rv(dev(F), dev(nu), dev(out[::-1].copy()), beta, 3.0).cpu().numpy()
    assert np.max(np.abs(back[::-1] / want - 1)) < 1e-11
    # <g, A F> = <A^T g, F>
    g = rng.standard_normal(n_out)
    gF, _ = xs.response_ip_rv_adjoint(dev(g), dev(F), dev(nu), dev(out), beta, 3.0)
    assert abs(gF.cpu().numpy() @ F - g @ want) <= 1e-11 * np.abs(g) @ want


@pytest.mark.parametrize("N,vsini,width", [(31, 40.0, 10.0), (129, 200.0, 10.0), (8200, 77.7, 10.0), (300, 9000.3, 2000.0)])
def test_rotation_against_the_oracle(xs, N, vsini, width):
    nu = 4360.0 * (1.0 + width / 4360.0) ** (np.arange(N) / (N - 1))
    F = spectrum(nu)
    want = oracle.rotation(F, nu, vsini, 0.45, 0.2)
    got = xs.response_rotation(dev(F), dev(nu), vsini, 0.45, 0.2).cpu().numpy()
    # the kernel's slope at its edges (up to ~10 a unit of x) on velocities good to 3e-11 km/s
    assert np.max(np.abs(got / want - 1)) < 1e-10
    g = np.random.default_rng(N).standard_normal(N)
    gF, _ = xs.response_rotation_adjoint(dev(g), dev(F), dev(nu), vsini, 0.45, 0.2)
    assert abs(gF.cpu().numpy() @ F - g @ want) <= 1e-10 * np.abs(g) @ want
