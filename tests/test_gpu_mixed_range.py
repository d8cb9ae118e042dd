"""Mixed precision where its FP32 forms could leave the range of FP32: lists of very wide
lines with lines of no width among them, low wavenumbers, against FP64, sums and adjoints, with the
tolerances of the other mixed cases (1e-5 of sigma above 1e-6 of a layer's largest, 1e-4 of
the largest gradient)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda")


def compare(lines, nu, T, P, cut, lam_of, sb=1.0):
    """lam_of(sigma): dF/dsigma from the FP64 sigma [L][N]."""
    from paper_2105_14782_gb300 import xs
    dl = xs.DeviceLines(lines)
    args = dl, dev(nu), dev(T), dev(P)
    want = xs.xs_compute(*args, sb, cut, xs.PREC_FP64)
    lam = lam_of(want)
    ref = [v.cpu().numpy() for v in xs.xs_compute_adjoint(*args, lam, sb, cut, xs.PREC_FP64)]
    big = max(np.max(np.abs(ref[0] * T)), abs(ref[1][0]))
    assert torch.isfinite(want).all() and np.isfinite(big)
    m = want > 1e-6 * want.amax(dim=1, keepdim=True)
    small = torch.empty(xs.lib().xs_workspace_min_bytes(dl.n, len(nu), len(T), xs.PREC_MIXED), dtype=torch.uint8,
                        device="cuda")
    for ws in (None, small):  # the full plan and the smallest accepted workspace
        got = xs.xs_compute(*args, sb, cut, xs.PREC_MIXED, workspace=ws).double()
        assert torch.isfinite(got).all()
        assert float(((got - want).abs() / want)[m].max()) < 1e-5
        g_T, g_b = (v.cpu().numpy() for v in xs.xs_compute_adjoint(*args, lam, sb, cut, xs.PREC_MIXED, workspace=ws))
        assert np.isfinite(g_T).all() and np.isfinite(g_b).all()
        assert np.max(np.abs(g_T - ref[0]) * T) <= 1e-4 * big and abs(g_b - ref[1])[0] <= 1e-4 * big


@pytest.mark.parametrize("nu0,every", [(1000.0, 40), (500.0, 40), (500.0, 7), (200.0, 40)])
def test_lines_without_width_among_wide_ones(nu0, every):
    """At 100 bar these lines are 1,700 to 8,500 Doppler widths wide (a); the ones without
    width need the near forms at the same points."""
    n, N = 2000, 2000
    lines = W.water_like(n, seed=int(nu0) + every, nu_min=nu0, nu_max=1.01 * nu0)
    lines.gamma_ref[:] = 0.1
    lines.gamma_ref[::every] = 0.0
    lines.ln_S0[1::every] += np.log(1e3)  # up to 1e-17 cm/molecule
    rng = np.random.default_rng(every)
    compare(lines, W.grid_lognu(N, nu0, 1.01 * nu0), np.array([700.0, 1000.0, 1000.0]), np.array([0.1, 30.0, 100.0]),
            0.003 * nu0, lambda s: (1.0 + 0.5 * dev(rng.uniform(size=(3, N)))) / s.amax(dim=1, keepdim=True))


@pytest.mark.parametrize("nu0,T0", [(7.69, 1000.0), (3.84, 500.0), (0.5, 300.0)])
@pytest.mark.parametrize("weight", [1e20, 1e25])
def test_low_wavenumbers(nu0, T0, weight):
    """Doppler widths go as the wavenumber, so 1/distance^2 reaches 1e7 cm^2 at these, its sixth
    power beyond FP32; weights of dF/dsigma as a well-measured spectrum gives them."""
    n, N = 1500, 2000
    lines = W.water_like(n, seed=5, nu_min=0.999 * nu0, nu_max=1.011 * nu0)
    lines.mass_amu = 28.0
    rng = np.random.default_rng(3)
    compare(lines, W.grid_lognu(N, nu0, 1.01 * nu0), np.array([0.8 * T0, T0, T0]), np.array([1e-6, 1e-4, 1e-3]),
            0.004 * nu0, lambda s: weight * (1.0 + 0.5 * dev(rng.uniform(size=(3, N)))))


@pytest.mark.parametrize("n,N,L", [(300, 40, 3), (3000, 2500, 5), (20000, 1500, 4)])
def test_weights_of_mixed_sign(n, N, L):
    """A fitted spectrum's dF/dsigma has both signs and its sums cancel.  An evaluation is good to
    1e-6 and the terms of dln sigma/dln T are up to ten times one (E'' c2/T of 5,000 cm^-1), so
    1e-5 of the sum of |lambda| sigma bounds T g_T and g_b (1e-3 to 1e-1 of what weights of one
    sign would give)."""
    from paper_2105_14782_gb300 import xs
    dl = xs.DeviceLines(W.water_like(n, seed=n))
    rng = np.random.default_rng(n)
    nu, P = W.grid_lognu(N), 10.0 ** np.linspace(-3, 2, L)
    args = dl, dev(nu), dev(1300.0 * P ** 0.1), dev(P)
    s = xs.xs_compute(*args, 1.1, 25.0, xs.PREC_FP64)
    lam = dev(rng.standard_normal((L, N))) / s.amax(dim=1, keepdim=True)
    size = (lam * s).abs().sum(dim=1)
    want = xs.xs_compute_adjoint(*args, lam, 1.1, 25.0, xs.PREC_FP64)
    got = xs.xs_compute_adjoint(*args, lam, 1.1, 25.0, xs.PREC_MIXED)
    assert torch.all((got[0] - want[0]).abs() * args[2] <= 1e-5 * size)
    assert abs((got[1] - want[1]).item()) <= 1e-5 * float(size.sum())
