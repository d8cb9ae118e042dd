"""FP64 leaves whose last point lies within rounding of |z| = 10 of a line, where the points
change from the wing polynomial to the series: the leaf and the point round the distance
differently, and either may be the one below 10."""
from fractions import Fraction

import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N, LEAF, T, P, MASS = 4096, 32, 1300.0, 1.0, 18.0
KB, AMU, CL = 1.380649e-16, 1.66053906660e-24, 2.99792458e10


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda")


def square(x, a2):  # fma(x, x, a2)
    return float(Fraction(x) ** 2 + Fraction(a2))


def edge_lines(nu):
    """Centres and widths (a = 0.02 .. 6) for which |z|^2 of a leaf's end point is 100 or more
    by the leaf's middle and half-width but below 100 by the point's own distance."""
    out = []
    for i in range(2, N // LEAF - 2):
        v0, v1 = float(nu[i * LEAF]), float(nu[i * LEAF + LEAF - 1])
        mid, h = 0.5 * (v0 + v1), 0.5 * (v1 - v0)
        for v, side in ((v0, -1.0), (v1, 1.0)):
            gamma = 1e-4 * 1.35 ** (i % 20)
            cen = v
            for _ in range(3):  # the distance at which |z| = 10, with the line's own constants
                c = 1.0 / (1.41421356237309504880 * (np.sqrt(KB * T / (MASS * AMU)) * cen / CL))
                a = gamma * (P / 1.01325) * c
                cen = v + side * np.sqrt(100.0 - a * a) / c
            for k in range(-3, 4):
                t = cen + k * np.spacing(cen)
                c = float(1.0 / (1.41421356237309504880 * (np.sqrt(KB * T / (MASS * AMU)) * t / CL)))
                a = gamma * (P / 1.01325) * c
                leaf = square(max(abs(mid - t) - h, 0.0) * c, a * a)
                if leaf >= 100.0 > square(abs(v - t) * c, a * a):
                    out.append((t, gamma))
    return np.array(out)


def test_leaf_ends_at_the_series_boundary():
    from paper_2105_14782_gb300 import xs
    nu = W.grid_lognu(N)
    e = edge_lines(nu)
    assert len(e) >= 20
    n = len(e)
    for extra in (0, 400):  # below and above the list length from which intervals are used
        filler = W.water_like(extra, seed=11)
        lines = W.LineList(np.append(e[:, 0], filler.nu_hat), np.append(np.full(n, np.log(1e-20)), filler.ln_S0),
                           np.append(np.zeros(n), filler.elower), np.append(e[:, 1], filler.gamma_ref),
                           np.append(np.zeros(n), filler.n_temp), MASS)
        lines = lines.subset(np.argsort(lines.nu_hat, kind="stable"))
        dl = xs.DeviceLines(lines)
        want = oracle.xs(lines, nu, [T], [P])
        got = xs.xs_compute(dl, dev(nu), dev([T]), dev([P]), prec=xs.PREC_FP64).cpu().numpy()
        assert np.max(np.abs(got - want) / want) < 1e-10
        # the adjoint of the leaves' end points, and the same on a grid without its first
        # points, whose leaves end elsewhere
        lam = np.zeros(N)
        lam[LEAF - 1::LEAF] = lam[::LEAF] = 1.0 / want[0].max()
        lam[:5] = 0.0
        g, s = (xs.xs_compute_adjoint(dl, dev(nu[q]), dev([T]), dev([P]), dev(lam[None, q]), prec=xs.PREC_FP64)
                for q in (slice(0, N), slice(5, N)))
        for u, v in zip(g, s):
            assert abs(u.item() - v.item()) <= 1e-10 * abs(v.item())
