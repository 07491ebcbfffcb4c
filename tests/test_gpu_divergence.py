"""The 2D divergence on both sides of the sizes where its derivatives change form (bands below 32 rows, both axes in
one launch, a launch per axis) against dense Pade matrices; tolerance: FP64 rounding of a sum of n^2 squares."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2306_17263_gb300 as pkg  # noqa: E402


def _pade(n, closure):
    """Node -> half-node derivative times h."""
    a = 22.0 * np.eye(n) + np.eye(n, k=1) + np.eye(n, k=-1)
    if closure == pkg.CLOSURE_PAPER:
        a[0] = a[-1] = 0.0
        a[0, :4] = [26.0, -5.0, 4.0, -1.0]
        a[-1, -4:] = a[0, 3::-1]
    else:
        a[0, 0] = a[-1, -1] = 23.0
    return np.linalg.solve(a / 24.0, np.eye(n, n + 1, k=1) - np.eye(n, n + 1))


@pytest.mark.parametrize("closure", [pkg.CLOSURE_PAPER, pkg.CLOSURE_REFLECT])
@pytest.mark.parametrize("precision", [pkg.FP64, pkg.FP32_REFINED])
@pytest.mark.parametrize("n", [5, 31, 32, 33, 64, 300, 770, 810])
def test_divergence(n, precision, closure):
    init = workloads.random_fields(n, seed=n)
    with pkg.Grid(n, 0.5, precision=precision, closure=closure) as g:
        g.set_fields(*init)
        _, hx, hy = g.get_fields()
        got = g.divergence()
    w = _pade(n, closure)
    want = np.linalg.norm((hx @ w.T + w @ hy) * n) / n
    assert abs(got - want) <= 1e-13 * n * want
