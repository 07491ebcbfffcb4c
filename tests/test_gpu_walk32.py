"""FP32_REFINED 2D steps at the sizes where the walking kernels change form: the smallest grids (explicit
rows up to 16 cells), strips of 112 and 120 columns ending inside, on and past a line's last columns,
segments of 16, 32 and 64 rows, and each number of solve levels (r).  Random fields against the FP64
oracle (FP64 GPU path for the large grid); tolerance as in the parity tests: FP32 noise of about 1e-7 per
step on grid-scale data."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2306_17263_gb300 as pkg  # noqa: E402


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("closure", [pkg.CLOSURE_PAPER, pkg.CLOSURE_REFLECT])
@pytest.mark.parametrize("n", [5, 6, 15, 16, 17, 18, 24, 31, 32, 33, 47, 64, 111, 112, 113, 114, 119, 120, 121, 122,
                               123, 126, 127, 128, 129, 225, 233, 241, 319, 320, 321, 345])
def test_steps_match_oracle(n, closure):
    r, steps = (0.3, 0.5, 0.65)[n % 3], 3
    o = oracle.Oracle2D(n, r, 1.3, closure)
    init = workloads.random_fields(n, seed=n)
    ref = [a.copy() for a in init]
    o.run(*ref, steps)
    with pkg.Grid(n, r, z=1.3, precision=pkg.FP32_REFINED, closure=closure) as g:
        g.set_fields(*init)
        g.run(steps)
        got = g.get_fields()
    for a, b in zip(got, ref):
        assert _rel(a, b) <= 2e-6
        assert np.all(a[b == 0.0] == 0.0)  # the walls of Dirichlet axes


@pytest.mark.parametrize("closure", [pkg.CLOSURE_PAPER, pkg.CLOSURE_REFLECT])
def test_long_segments(closure):
    n, r, steps = 1801, 0.5, 2
    init = workloads.random_fields(n, seed=7)
    out = []
    for precision in (pkg.FP64, pkg.FP32_REFINED):
        with pkg.Grid(n, r, precision=precision, closure=closure) as g:
            g.set_fields(*init)
            g.run(steps)
            out.append(g.get_fields())
    for a, b in zip(*out):
        assert _rel(b, a) <= 2e-6


def test_batch_cavities_equal_single_grids():
    sizes = [5, 16, 17, 65, 113, 121, 330, 345]
    with pkg.Batch(sizes, 0.5) as b:
        for c, n in enumerate(sizes):
            b.set_fields(c, *workloads.random_fields(n, seed=n))
        b.run(3)
        got = [b.get_fields(c) for c in range(len(sizes))]
    for n, fields in zip(sizes, got):
        with pkg.Grid(n, 0.5, precision=pkg.FP32_REFINED) as g:
            g.set_fields(*workloads.random_fields(n, seed=n))
            g.run(3)
            for a, e in zip(fields, g.get_fields()):
                assert np.array_equal(a, e)


@pytest.mark.parametrize("closure", [pkg.CLOSURE_PAPER, pkg.CLOSURE_REFLECT])
@pytest.mark.parametrize("n", [5, 31, 32, 33, 34, 47, 64, 65, 103, 104, 105, 116, 117, 118, 127, 128, 129, 130, 209,
                               233, 260])
def test_reverse_steps_match_oracle(n, closure):
    """The walking reverse pass: end segments, strips of 104 columns, FP64 below 32 cells."""
    r, steps = (0.3, 0.5, 0.65)[n % 3], 3
    o = oracle.Oracle2D(n, r, 1.3, closure)
    lam = workloads.random_fields(n, seed=n + 1)
    ref = [a.copy() for a in lam]
    for _ in range(steps):
        o.step_T(*ref)
    with pkg.Grid(n, r, z=1.3, precision=pkg.FP32_REFINED, closure=closure) as g:
        got = g.adjoint_steps(steps, *lam)
    for a, b in zip(got, ref):
        assert _rel(a, b) <= 2e-6
