"""The x-z stage kernel at the edges of its tiles (64 or 32 columns by 14 or 28 rows: one less, one
more, the fewest cells), against the oracle over two steps with the parity suite's bounds (1e-12 in
FP64, 1e-5 in FP32, relative L2 per field), for every tile shape; and the tile-to-domain search on
more domains than a warp takes at once, bitwise against each domain alone."""
import numpy as np
import pytest

import workloads as W
from oracle import Oracle

from test_gpu_parity import TOL, rel_errs, rounded

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_02955_gb300 import build
    build.build()


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("kind", ["viscous", "moist"])
@pytest.mark.parametrize("n", [(3, 15), (33, 3), (31, 14), (65, 29), (64, 28), (129, 13)])
def test_plane_tiles_against_the_oracle(kind, dtype, n):
    from paper_1901_02955_gb300 import Context
    if kind == "viscous":
        w = W.add_random_motion(W.density_current(nx=n[0], nz=n[1], dtype=dtype))
    else:
        w = W.add_random_motion(W.moist_bubble(nx=n[0], nz=n[1], dtype=dtype))
    Y0 = rounded(w, dtype)
    ctx = Context(w, dtype=dtype)
    ctx.set_state(Y0)
    dt = ctx.compute_dt()
    want, _, rc = Oracle(w).step(Y0, 2, dt=dt)
    assert rc == 0
    for v in range(ctx.info()["n_tile_variants"]):
        ctx.set_tile_variant(v)
        ctx.set_state(Y0)
        ctx.step(2, dt_fixed=dt)
        err = rel_errs(ctx.get_state(), want, Y0, w)
        assert max(err) <= TOL[dtype], (v, err)
    ctx.close()


def test_many_domains_each_equal_to_its_own_context():
    from paper_1901_02955_gb300 import Context
    ws = [W.add_random_motion(W.warm_bubble(n=3 + (7 * i) % 40), seed=W.BASE_SEED + i)
          for i in range(70)]
    ctx = Context(ws, dtype="f64")
    ctx.set_tile_variant(1)
    for d, w in enumerate(ws):
        ctx.set_state(w.Y, domain=d)
    ctx.step(2)
    for d, w in enumerate(ws):
        one = Context(w, dtype="f64")
        one.set_tile_variant(1)
        one.set_state(w.Y)
        one.step(2)
        assert np.array_equal(ctx.get_state(domain=d), one.get_state()), d
        one.close()
    ctx.close()
