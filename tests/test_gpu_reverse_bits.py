"""Accuracy of the FP32 reverse pass against the FP64 one: the phase of one mode over tens of thousands of transposed
steps, where a coherent error of a coefficient or of a line's ends grows, and the rounding of a single step.
_bound, relative to omega T: 1e-10, the error the solve's polynomial is built to, and about sixteen roundings of
2^-24 per point and step, independent over points and steps; with_rho adds what rho as an FP32 number (off by
1.1e-9) does to a derivative at theta = pi k / n."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2306_17263_gb300 as pkg  # noqa: E402


def _both(n, r, z, closure, steps, state):
    out = []
    for precision in (pkg.FP64, pkg.FP32_REFINED):
        with pkg.Grid(n, r, z=z, precision=pkg.FP32_REFINED, closure=closure) as g:
            g.set_adjoint_precision(precision)
            out.append(g.adjoint_steps(steps, *state))
    return out


def _shift(n, r, k, steps, closure, z):
    x = np.pi * k * np.arange(n + 1) / n
    s, c = np.sin(x), np.cos(np.pi * k * (np.arange(n) + 0.5) / n)
    ee, eh = np.outer(s, s), np.outer(c, s)
    ph = []
    for e, hx, hy in _both(n, r, z, closure, steps, (ee, np.zeros_like(eh), np.zeros_like(eh.T))):
        h = (np.sum(hy * eh.T) - np.sum(hx * eh)) / np.sum(eh ** 2)
        ph.append(math.atan2(h / (z * math.sqrt(2.0)), np.sum(e * ee) / np.sum(ee ** 2)))
    d = (ph[1] - ph[0] + math.pi) % (2.0 * math.pi) - math.pi
    return abs(d) / (math.pi * k * math.sqrt(2.0) * steps * r / n)


def _bound(n, k, steps, with_rho=False):
    return (1e-10 + (2e-9 * (math.pi * k / n) ** 2 if with_rho else 0.0)
            + 16.0 * 2.0 ** -24 / ((n - 1) * math.sqrt(steps)))


CLOSURES = [pkg.CLOSURE_PAPER, pkg.CLOSURE_REFLECT]


@pytest.mark.parametrize("closure", CLOSURES)
@pytest.mark.parametrize("n, r, k, steps", [(33, 0.65, 3, 40000), (128, 0.65, 4, 20000)])
def test_line_ends(n, r, k, steps, closure):
    assert _shift(n, r, k, steps, closure, 1.0) <= _bound(n, k, steps, with_rho=True)


@pytest.mark.parametrize("n, r, k, z", [(32, 0.5, 10, 1.0), (32, 0.5, 10, 1.3), (64, 0.68, 20, 1.0), (64, 0.65, 12, 1.3)])
def test_filter_coefficients(n, r, k, z):
    """Short waves: rho of the recurrences, s and 12 beta s of the filter."""
    assert _shift(n, r, k, 40000, pkg.CLOSURE_REFLECT, z) <= _bound(n, k, 40000)


@pytest.mark.parametrize("closure", CLOSURES)
@pytest.mark.parametrize("n, r", [(700, 0.3), (700, 0.68), (1024, 0.5), (1024, 0.65)])
def test_one_step_rounds_the_derivative_once(n, r, closure):
    """The H fields one transposed step makes of a smooth E_z: one rounding of the derivative, 0.4 * 2^-24 of its
    RMS, and as much again in square from all else, away from the walls."""
    rng = np.random.default_rng(n)
    k = np.arange(1, 13)
    s = np.sin(np.pi * np.outer(np.arange(n + 1), k) / n)
    e = s @ rng.standard_normal((k.size, k.size)) @ s.T
    e[0] = e[-1] = e[:, 0] = e[:, -1] = 0.0
    want, got = _both(n, r, 1.0, closure, 1, (e, np.zeros((n, n + 1)), np.zeros((n + 1, n))))
    for a, b in zip(want[1:], got[1:]):
        a, b = a[32:-32, 32:-32], b[32:-32, 32:-32]
        assert np.linalg.norm(b - a) <= math.sqrt(2.0) * 0.4 * 2.0 ** -24 * np.linalg.norm(a)
