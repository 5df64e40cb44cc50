"""A record's last segment comes from the forward run itself: the adjoint after it, the same adjoint
asked for again (its segments are recomputed by then) and adjoints of other step counts and
checkpoint spacings in the same context (the record's memory is used again) all equal, bitwise, the
adjoint of a fresh context that keeps every stage input."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_02955_gb300 import build
    build.build()


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("moist", [False, True])
def test_adjoint_after_reused_records(dtype, moist):
    from paper_1901_02955_gb300 import Context
    make = W.moist_adjoint_bubble if moist else W.warm_bubble
    w = W.add_random_motion(make(n=33, dtype=dtype))
    lam = np.random.default_rng(3).standard_normal(w.Y.shape)

    def reference(n):
        ctx = Context(w, dtype=dtype)
        ctx.set_state(w.Y)
        ctx.record(n, 0)
        out = ctx.step_adjoint(n, lam), ctx.get_state()
        ctx.close()
        return out

    want = {n: reference(n) for n in (1, 5, 7)}
    ctx = Context(w, dtype=dtype)
    for n, every in [(7, 3), (7, 7), (5, 1), (1, 4), (7, 2), (5, 8), (7, 3)]:
        ctx.set_state(w.Y)
        ctx.record(n, every)
        for again in range(2):
            assert np.array_equal(ctx.step_adjoint(n, lam), want[n][0]), (n, every, again)
            assert np.array_equal(ctx.get_state(), want[n][1]), (n, every, again)
    ctx.close()
