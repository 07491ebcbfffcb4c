"""FP64 line recurrences and polynomial solves at the sizes where they change form: the shortest lines
they take (below that, explicit bands), segments of 16 and 32 rows ending inside, on and past a line's
last rows, tiles of 8 and 16 points and the level-by-level solve of large grids.  Tolerances as in the
operator parity tests (rounding of ~40 operations per point, truncations below 1e-16)."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2306_17263_gb300 as pkg  # noqa: E402


def _dev(a):
    return torch.tensor(a, device="cuda")


@pytest.mark.parametrize("closure", [pkg.CLOSURE_PAPER, pkg.CLOSURE_REFLECT])
@pytest.mark.parametrize("n", [31, 32, 33, 34, 47, 48, 49, 63, 64, 65, 66, 161, 200, 201, 390, 545, 560])
def test_curls_and_solves(n, closure):
    r = 0.5
    o = oracle.Oracle2D(n, r, closure=closure)
    ez, hx, hy = workloads.random_fields(n, seed=n)
    with pkg.Grid(n, r, closure=closure) as g:
        R, Rx, Ry = (torch.full(s, 7.0, dtype=torch.float64, device="cuda") for s in g.shapes())
        g.apply_op("curl_he", [_dev(hx), _dev(hy)], [R])
        g.apply_op("curl_eh", [_dev(ez)], [Rx, Ry])
        g.sync()
        for got, ref in zip((R, Rx, Ry), (o.curl_h_to_e(hx, hy), *o.curl_e_to_h(ez))):
            assert np.max(np.abs(got.cpu().numpy() - ref)) <= 1e-13 * np.max(np.abs(ref))
        for f, (name, u) in enumerate((("ez", ez), ("hx", hx), ("hy", hy))):
            x_ref, _ = o.p1_solve(f, u)
            out = torch.full(u.shape, 7.0, dtype=torch.float64, device="cuda")
            g.apply_op(f"p1solve_{name}", [_dev(u)], [out])
            inplace = _dev(u)
            g.apply_op(f"p1solve_{name}", [inplace], [inplace])
            g.sync()
            assert np.max(np.abs(out.cpu().numpy() - x_ref)) <= 1e-12 * np.max(np.abs(x_ref))
            assert torch.equal(inplace, out)


@pytest.mark.parametrize("closure", [pkg.CLOSURE_PAPER, pkg.CLOSURE_REFLECT])
@pytest.mark.parametrize("n", [31, 32, 33, 49, 66, 131])
def test_adjoint_step_is_the_transpose(n, closure):
    """<M u, v> = <u, M^T v>, and M^T v against the oracle's reverse step."""
    o = oracle.Oracle2D(n, 0.5, closure=closure)
    u, v = workloads.random_fields(n, seed=1), workloads.random_fields(n, seed=2)
    ref = [a.copy() for a in v]
    o.step_T(*ref)
    with pkg.Grid(n, 0.5, closure=closure) as g:
        g.set_fields(*u)
        g.step()
        mu = g.get_fields()
        mv = g.adjoint_steps(1, *v)
    for a, b in zip(mv, ref):
        assert np.linalg.norm(a - b) <= 1e-12 * np.linalg.norm(b)
    x, y = sum(np.vdot(a, b) for a, b in zip(mu, v)), sum(np.vdot(a, b) for a, b in zip(u, mv))
    scale = np.sqrt(sum(np.vdot(a, a) for a in mu) * sum(np.vdot(a, a) for a in v))
    assert abs(x - y) <= 1e-12 * scale


@pytest.mark.parametrize("closure", [pkg.CLOSURE_PAPER, pkg.CLOSURE_REFLECT])
@pytest.mark.parametrize("n", [32, 33, 35, 50])
def test_3d_step(n, closure):
    init = workloads.random_fields3(n, seed=n)
    o = oracle.Oracle3D(n, 0.4, Z=1.3, closure=closure)
    ref = [a.copy() for a in init]
    o.run(ref, 1)
    with pkg.Grid(n, 0.4, z=1.3, closure=closure, dim=3) as g:
        g.set_fields(*init)
        g.step()
        got = g.get_fields()
    for a, b in zip(got, ref):
        assert np.linalg.norm(a - b) <= 1e-12 * np.linalg.norm(b)


@pytest.mark.parametrize("n", [31, 32, 33, 64, 546, 547, 764, 800])
def test_2d_steps_at_launch_limits(n):
    """Both derivatives of a half-step in one launch, and the two terms of Step 1 summed by the solve, up to
    the sizes where the solve's levels (547) and then the derivatives (about 780) take launches of their own."""
    r, steps = 0.5, 2
    o = oracle.Oracle2D(n, r)
    init = workloads.random_fields(n, seed=n)
    ref = [a.copy() for a in init]
    o.run(*ref, steps)
    with pkg.Grid(n, r) as g:
        g.set_fields(*init)
        g.run(steps)
        got = g.get_fields()
    for a, b in zip(got, ref):
        assert np.linalg.norm(a - b) <= 1e-12 * np.linalg.norm(b)
        assert np.all(a[b == 0.0] == 0.0)
