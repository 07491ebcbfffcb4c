"""Coefficients of the FP32_REFINED step over long runs: the phase of one cavity mode after tens of thousands of
steps against the FP64 step.  A coefficient that is off by a relative eps shifts the frequency by about eps, the
same way in every step, where rounding averages out; so does a small term that rounds away in every sum.  _bound is
what may remain, relative to omega T:
  1e-10            the error the solve's polynomial is built to
  + 2e-9 theta^2   rho of the recurrences as an FP32 number (off by 1.9e-9 at most, its gain exact at theta = 0),
                   theta = pi k / n
  + 16 * 2^-24 / ((n - 1) sqrt(steps))   about sixteen roundings per point and step, independent over points and
                   steps."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2306_17263_gb300 as pkg  # noqa: E402


def _phase(fields, n, k, z):
    x = np.pi * k * np.arange(n + 1) / n
    s, c = np.sin(x), np.cos(np.pi * k * (np.arange(n) + 0.5) / n)
    ez, hx, hy = fields
    e = np.sum(ez * np.outer(s, s)) / np.sum(np.outer(s, s) ** 2)
    b = np.sum(np.outer(c, s) ** 2)
    h = (np.sum(hy * np.outer(s, c)) - np.sum(hx * np.outer(c, s))) / b
    return math.atan2(h * z / math.sqrt(2.0), e)


def _shift(n, r, k, steps, closure, z=1.3):
    ph = []
    for precision in (pkg.FP64, pkg.FP32_REFINED):
        with pkg.Grid(n, r, z=z, precision=precision, closure=closure) as g:
            g.init_modes([(k, k, 1.0)])
            g.run(steps)
            ph.append(_phase(g.get_fields(), n, k, z))
    d = (ph[1] - ph[0] + math.pi) % (2.0 * math.pi) - math.pi
    return abs(d) / (math.pi * k * math.sqrt(2.0) * steps * r / n)


def _bound(n, k, steps):
    return 1e-10 + 2e-9 * (math.pi * k / n) ** 2 + 16.0 * 2.0 ** -24 / ((n - 1) * math.sqrt(steps))


CLOSURES = [pkg.CLOSURE_PAPER, pkg.CLOSURE_REFLECT]


@pytest.mark.parametrize("closure", CLOSURES)
@pytest.mark.parametrize("n, r, k", [(8, 0.5, 2), (16, 0.5, 3), (16, 0.65, 2)])
def test_smallest_grids_scale(n, r, k, closure):
    """Grids of at most 16 cells, whose derivatives come from explicit rows: no factor common to all of them is off
    by half an FP32 ulp."""
    assert _shift(n, r, k, 8000, closure) <= 2.0 ** -25


@pytest.mark.parametrize("closure", CLOSURES)
@pytest.mark.parametrize("n, r, k", [(6, 0.5, 1), (8, 0.5, 2), (12, 0.5, 2), (16, 0.5, 3), (16, 0.65, 2)])
def test_smallest_grids(n, r, k, closure):
    """The same grids: the rows' sums lose none of their small terms."""
    assert _shift(n, r, k, 20000, closure) <= _bound(n, k, 20000)


@pytest.mark.parametrize("closure", CLOSURES)
@pytest.mark.parametrize("n, r, k", [(17, 0.5, 2), (20, 0.5, 2), (32, 0.5, 3)])
def test_line_ends(n, r, k, closure):
    """Short lines of the walks: the closure's end rows."""
    assert _shift(n, r, k, 40000, closure) <= _bound(n, k, 40000)


@pytest.mark.parametrize("n, q, k, z", [(64, 96, 4, 1.0), (64, 52, 4, 1.0), (128, 52, 4, 1.3), (256, 57, 8, 1.0),
                                        (256, 57, 8, 1.3)])
def test_level_coefficients(n, q, k, z):
    """The solve's levels at r = sqrt(24 / q), where the filter's coefficient 12 + 24 / r^2 is a whole number; they
    weigh most near the stability limit."""
    assert _shift(n, math.sqrt(24.0 / q), k, 40000, pkg.CLOSURE_REFLECT, z) <= _bound(n, k, 40000)


@pytest.mark.parametrize("n, r, k, z", [(17, 0.65, 2, 1.3), (32, 0.68, 3, 1.0), (64, 0.68, 4, 1.3), (128, 0.68, 4, 1.0),
                                        (256, 0.65, 8, 1.0), (256, 0.65, 8, 1.3)])
@pytest.mark.parametrize("closure", CLOSURES)
def test_filter_coefficient(n, r, k, z, closure):
    """12 beta not exact in FP32."""
    assert _shift(n, r, k, 40000, closure, z) <= _bound(n, k, 40000)


def _shift3(n, r, steps, closure, z=1.3):
    """The same in 3D for the mode (2, 1, 2): E and H projected on their own shapes at the start."""
    w = 3.0 * math.pi
    ph = []
    for precision in (pkg.FP64, pkg.FP32_REFINED):
        with pkg.Grid(n, r, z=z, precision=precision, closure=closure, dim=3) as g:
            g.init_modes([(2, 1, 2, 1.0, 0.0, -1.0)])
            s = g.get_fields()
            g.run(steps)
            f = g.get_fields()
        e, h = (sum(np.sum(a * b) for a, b in zip(f[q], s[q])) / sum(np.sum(b * b) for b in s[q])
                for q in (slice(0, 3), slice(3, 6)))
        ph.append(math.atan2(h * math.sin(0.5 * w * r / n), e))
    d = (ph[1] - ph[0] + math.pi) % (2.0 * math.pi) - math.pi
    return abs(d) / (w * steps * r / n)


def _bound3(n, steps):
    return 1e-10 + 2e-9 * (2.0 * math.pi / n) ** 2 + 16.0 * 2.0 ** -24 / ((n - 1) ** 1.5 * math.sqrt(steps))


@pytest.mark.parametrize("closure", CLOSURES)
@pytest.mark.parametrize("n, r", [(17, 0.4), (20, 0.3), (24, 0.4)])
def test_line_ends_3d(n, r, closure):
    assert _shift3(n, r, 10000, closure) <= _bound3(n, 10000)


@pytest.mark.parametrize("r, z", [(0.515, 2.0), (0.54, 1.0), (0.55, 1.0)])
def test_level_coefficients_3d(r, z):
    """Where the last level's coefficient and the increment scale are farthest from FP32 numbers."""
    assert _shift3(64, r, 4000, pkg.CLOSURE_REFLECT, z) <= _bound3(64, 4000)
