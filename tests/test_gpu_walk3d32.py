"""FP32_REFINED 3D steps at the sizes where the kernels change form: lines too short for the walks, strips
of 32 columns and marches of 16 planes ending inside, on and past a component's last points, one and several
segments per line.  Random fields against the FP64 oracle (FP64 GPU path for the larger grids); tolerance as
in the parity tests: FP32 noise of about 1e-7 per step on grid-scale data."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2306_17263_gb300 as pkg  # noqa: E402


def _run(n, r, closure, precision, init, steps):
    with pkg.Grid(n, r, precision=precision, closure=closure, dim=3) as g:
        g.set_fields(*init)
        g.run(steps)
        return g.get_fields()


@pytest.mark.parametrize("closure", [pkg.CLOSURE_PAPER, pkg.CLOSURE_REFLECT])
@pytest.mark.parametrize("n", [5, 8, 15, 16, 17, 18, 19, 24, 31, 32, 33, 34, 35, 47, 49, 63, 64, 65, 66, 67, 97, 131])
def test_steps_match(n, closure):
    r, steps = (0.2, 0.4, 0.5)[n % 3], 2
    init = workloads.random_fields3(n, seed=n)
    got = _run(n, r, closure, pkg.FP32_REFINED, init, steps)
    if n <= 34:
        o = oracle.Oracle3D(n, r, closure=closure)
        ref = [a.copy() for a in init]
        o.run(ref, steps)
    else:
        ref = _run(n, r, closure, pkg.FP64, init, steps)
    for a, b in zip(got, ref):
        assert np.linalg.norm(a - b) <= 2e-6 * np.linalg.norm(b)
        assert np.all(a[b == 0.0] == 0.0)  # the walls of Dirichlet axes
