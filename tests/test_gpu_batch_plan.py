"""A launch plan that cannot be applied (its work lists fail to allocate, by host-side injection) leaves the
batch as it was: the old plan, its lists and the graphs captured from them stay in use."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2306_17263_gb300 as pkg  # noqa: E402

SIZES = [8, 24, 40]


def _run(fail_at):
    with pkg.Batch(SIZES, 0.5) as b:
        for k, n in enumerate(SIZES):
            b.set_fields(k, *workloads.random_fields(n, seed=40 + k))
        b.run(20)  # captures the graphs of the plan in use
        if fail_at:
            plan, held = b.plan(), pkg.debug_live_allocs()
            try:
                pkg.debug_fail_alloc(fail_at)
                with pytest.raises(pkg.MaxwellError) as e:
                    b.set_plan(2 if plan[0] != 2 else 0, plan[1], plan[2])
            finally:
                pkg.debug_fail_alloc(0)
            assert e.value.status == -3
            assert b.plan() == plan
            assert pkg.debug_live_allocs() == held
        b.run(17)
        b.step()
        return [b.get_fields(k) for k in range(len(SIZES))]


@pytest.mark.parametrize("fail_at", [1, 2, 3, 4])
def test_failed_plan_leaves_the_batch_as_it_was(fail_at):
    for got, want in zip(_run(fail_at), _run(0)):
        for a, c in zip(got, want):
            assert np.array_equal(a, c)
