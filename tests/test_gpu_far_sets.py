"""Line sums where the split into near and far lines can go wrong: grids of one point, of
part of a leaf and just over an interval's end, grids with gaps, wing cuts from below a
Doppler width to the whole band, lists on both sides of the length from which the far
lines are taken at interval nodes."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def xs():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2105_14782_gb300 import xs as _xs
    return _xs


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda")


def grid(kind, N, rng):
    if kind == "log":
        return W.grid_lognu(N, 4360.0, 4370.0)
    if kind == "random":
        return np.sort(rng.uniform(4360.0, 4370.0, N))
    return np.sort(np.concatenate([rng.uniform(4360.0, 4360.3, N // 2), rng.uniform(4369.0, 4370.0, N - N // 2)]))


CASES = [("log", 1, 300, 25.0), ("log", 31, 256, 25.0), ("log", 33, 255, 25.0), ("log", 129, 1000, 3.0),
         ("log", 2049, 3000, 25.0), ("log", 2048, 700, 0.01), ("random", 513, 2000, 2.0), ("gaps", 700, 2000, 4.0),
         ("log", 8200, 1500, 6.0),
         # on both sides of the density from which intervals are halved, not quartered
         ("log", 2049, 2 * 2049 - 1, 2.0), ("log", 2049, 2 * 2049, 2.0), ("log", 2300, 1149, 3.0), ("log", 2300, 1150, 3.0),
         ("gaps", 700, 6000, 4.0), ("random", 70, 3000, 1.0)]
P = np.array([1e-3, 0.3, 30.0])
T = np.array([700.0, 1200.0, 1900.0])


@pytest.mark.parametrize("kind,N,n,cut", CASES)
def test_sigma_against_the_oracle(xs, kind, N, n, cut):
    nu = grid(kind, N, np.random.default_rng(N))
    lines = W.water_like(n, seed=n, nu_min=4355.0, nu_max=4375.0)
    want = oracle.xs(lines, nu, T, P, sb=1.3, wing_cut=cut)
    dl = xs.DeviceLines(lines)
    m = want > 1e-6 * want.max(axis=1, keepdims=True)
    for prec, tol in ((xs.PREC_FP64, 1e-10), (xs.PREC_MIXED, 1e-5)):
        small = torch.empty(xs.lib().xs_workspace_min_bytes(n, N, 3, prec), dtype=torch.uint8, device="cuda")
        for ws in (None, small):  # the full plan and the smallest accepted workspace
            got = xs.xs_compute(dl, dev(nu), dev(T), dev(P), 1.3, cut, prec, workspace=ws).double().cpu().numpy()
            assert np.all((got == 0) == (want == 0))
            assert m.sum() == 0 or np.max(np.abs(got - want)[m] / want[m]) < tol


@pytest.mark.parametrize("kind,N,n,cut", CASES)
def test_adjoint_with_and_without_far_sets(xs, kind, N, n, cut):
    """FP64: the adjoint on the full plan (far lines at nodes) against the smallest workspace
    (every line point by point), the same sums in another order: 1e-10 of the sum of the
    terms' magnitudes, here bounded by that of a layer's largest gradient; mixed against
    FP64: 1e-4."""
    nu = grid(kind, N, np.random.default_rng(N))
    dl = xs.DeviceLines(W.water_like(n, seed=n, nu_min=4355.0, nu_max=4375.0))
    lam = dev(1e20 * (1.0 + 0.5 * np.random.default_rng(7).uniform(size=(3, N))))
    out = {}
    for prec in (xs.PREC_FP64, xs.PREC_MIXED):
        small = torch.empty(xs.lib().xs_workspace_min_bytes(n, N, 3, prec), dtype=torch.uint8, device="cuda")
        for name, ws in (("full", None), ("small", small)):
            g_T, g_b = xs.xs_compute_adjoint(dl, dev(nu), dev(T), dev(P), lam, 1.3, cut, prec, workspace=ws)
            out[prec, name] = np.append(g_T.cpu().numpy() * T, g_b.cpu().numpy())
    ref = out[xs.PREC_FP64, "small"]
    big = np.max(np.abs(ref))
    assert np.max(np.abs(out[xs.PREC_FP64, "full"] - ref)) <= 1e-10 * big
    for name in ("full", "small"):
        assert np.max(np.abs(out[xs.PREC_MIXED, name] - ref)) <= 1e-4 * big


@pytest.mark.parametrize("n,N", [(650, 6755), (1516, 2472)])
def test_fp64_nodes_keep_the_precision(xs, n, N):
    """FP64: far lines at nodes against every line at every point, few lines in narrow
    intervals over a wide band (where a node's position, rounded to an ulp of nu, would be
    1e-12 of an interval off): each is within about 1e-14 of the exact sum (the strengths'
    exponents, the same in both), so 3e-14 of each other."""
    nu, L = W.grid_lognu(N), 2
    dl = xs.DeviceLines(W.water_like(n, seed=n))
    p, t = dev([1e-3, 100.0]), dev([900.0, 1700.0])
    small = torch.empty(xs.lib().xs_workspace_min_bytes(n, N, L, xs.PREC_FP64), dtype=torch.uint8, device="cuda")
    a = xs.xs_compute(dl, dev(nu), t, p, 1.0, 25.0, xs.PREC_FP64)
    b = xs.xs_compute(dl, dev(nu), t, p, 1.0, 25.0, xs.PREC_FP64, workspace=small)
    m = b > 0
    assert float(((a - b).abs()[m] / b[m]).max()) < 3e-14
