"""Launches of one FP64 step: ms_launches_per_step and the events of ms_step_profiled, where a solve runs all
its levels in one launch and where each level is a launch of its own (more than 3e5 points of its fields
together), with the bytes a launch must touch."""
import math

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2306_17263_gb300 as pkg  # noqa: E402


def _degree(r, c, s, d):
    """Smallest m >= 2 with 1 / T_m((D - c) / s) <= 1e-17, D = 6 c1 h^2 + d."""
    x = (6.0 * 24.0 / r ** 2 * (1.0 + 2.0 / r ** 2) + d - c) / s
    m = 2
    while math.cosh(m * math.acosh(x)) < 1e17:
        m += 1
    return m


def _profile(n, r, dim, kind):
    with pkg.Grid(n, r, precision=pkg.FP64, dim=dim) as g:
        launches = g.launches_per_step
        rec = g.step_profiled()
    assert len(rec) == launches
    return [b for k, _, b in rec if k == kind]


@pytest.mark.parametrize("n, e_levels, h_levels", [(64, 0, 0), (386, 0, 0), (387, 0, 1), (546, 0, 1), (547, 1, 1),
                                                   (1024, 1, 1)])
@pytest.mark.parametrize("r", [0.3, 0.5, 0.65])
def test_2d_solves(n, e_levels, h_levels, r):
    m = _degree(r, 20.0, 16.0, 36.0)
    got = _profile(n, r, 2, "p1sweep64")
    want = []
    for levels, pts in ((e_levels, (n + 1) ** 2), (h_levels, 2 * n * (n + 1))):
        if levels:
            want += [8.0 * pts * q for q in [2] + [3] * (m - 3) + [4]]
        else:
            want.append(8.0 * pts * (4 if not want else 3))  # Step 1 reads two right-hand sides
    assert len(got) == len(want)
    assert got == want


@pytest.mark.parametrize("r", [0.3, 0.5])
def test_3d_solves(r):
    n, m = 12, _degree(r, 8.0, 16.0, 24.0)
    got = _profile(n, r, 3, "sweep3d64")
    pts = [3 * n * (n + 1) ** 2, 3 * n * n * (n + 1)]
    assert got == [8.0 * p * q for p in pts for q in [2] + [3] * (m - 3) + [4]]
