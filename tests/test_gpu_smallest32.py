"""FP32_REFINED on grids of at most 16 cells (explicit rows, two lines per warp) in the forms that differ from the
plain step: current sources, wall sources and the tracked Delta E, a few steps of random fields against the FP64
step; tolerance as in the parity tests: FP32 noise of about 1e-7 per step on grid-scale data."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2306_17263_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("form", ["sources", "wall sources", "tracked"])
@pytest.mark.parametrize("n", [5, 6, 8, 9, 15, 16, 17])
def test_forms_match_fp64(n, form):
    scheme = pkg.SCHEME_C4_DE if form == "tracked" else pkg.SCHEME_C4
    out = []
    for precision in (pkg.FP64, pkg.FP32_REFINED):
        with pkg.Grid(n, 0.5, z=1.3, precision=precision, scheme=scheme) as g:
            if form == "sources":
                g.set_sources([(1, 2, 0.7, 3.0), (2, 1, -0.4, 5.0)])
            elif form == "wall sources":
                g.set_sources_xy([(1, 2, 0.7, 3.0, 1, 0), (2, 1, -0.4, 5.0, 0, 1)])
            g.set_fields(*workloads.random_fields(n, seed=n))
            g.run(3)
            out.append(g.get_fields())
    for a, b in zip(*out):
        assert np.linalg.norm(b - a) <= 2e-6 * np.linalg.norm(a)
