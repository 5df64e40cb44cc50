"""The resident step takes every grid whose tiles are co-resident at the full height of the tile shape,
also where the height picked for three launches gives more tiles than that (a little more than one
wave), and the moist FP64 layout with two tiles per SM. It equals three launches there (bitwise, with
the saturation adjustment to 1e-6 of each field's largest value as in the other launch-mode tests),
and the tiling for three launches is back when the mode is left. In the other modes the heights do not
spill a few tiles into another round."""
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


def dry(nx, nz):
    return W.add_random_motion(W.density_current(nx=nx, nz=nz, nu=0.0))


def moist(nx, nz):
    return W.add_random_motion(W.moist_bubble(nx=nx, nz=nz))


@pytest.mark.parametrize("make,dtype,nx,nz,variant", [
    (dry, "f32", 336, 504, None), (dry, "f32", 768, 256, None), (dry, "f32", 1019, 153, None),
    (dry, "f32", 388, 497, 2), (dry, "f32", 795, 294, 1), (dry, "f32", 336, 504, 3),
    (dry, "f64", 544, 160, None), (dry, "f64", 381, 313, 0), (dry, "f64", 664, 172, 1),
    (moist, "f64", 483, 257, None), (moist, "f64", 436, 102, None), (moist, "f64", 698, 141, None),
    (moist, "f32", 560, 135, 1)])
def test_resident_step_takes_what_fits_at_full_height(make, dtype, nx, nz, variant):
    from paper_1901_02955_gb300 import Context
    w = make(nx, nz)
    ctx = Context(w, dtype=dtype)
    if variant is not None:
        ctx.set_tile_variant(variant)
    before = ctx.info()["tile"]
    out = []
    for mode in (0, 2, 0):
        ctx.use_persistent(mode)
        ctx.set_state(w.Y)
        ctx.step(3)
        out.append(ctx.get_state())
        assert ctx.info()["persistent"] == mode
    assert ctx.info()["tile"] == before
    ctx.close()
    scale = np.abs(out[0]).reshape(w.nv, -1).max(axis=1)
    for o in out[1:]:
        d = np.abs(o - out[0]).reshape(w.nv, -1).max(axis=1)
        assert np.all(d <= (1e-6 if make is moist else 0.0) * scale), d / scale


def test_resident_step_keeps_class_shapes_and_follows_a_change_of_shape():
    """Modes 0 and 2 in turn, a new shape in mode 2 (its tiles are cut for the resident step at the
    next step) and the size classes' own shapes, which mode 2 leaves alone."""
    from paper_1901_02955_gb300 import Context
    ws = [dry(336, 400), dry(100, 90)]
    ctx = Context(ws, dtype="f32")

    def advance():
        for d, w in enumerate(ws):
            ctx.set_state(w.Y, domain=d)
        ctx.step(2)
        return [ctx.get_state(domain=d) for d in range(2)]

    want = advance()
    ctx.set_class_tile_variant(0, 1)
    ctx.use_persistent(2)
    got = [advance()]
    assert ctx.info()["classes"][0]["variant"] == 1 and ctx.info()["per_class_tiles"] == 1
    ctx.use_persistent(0)
    got.append(advance())
    assert ctx.info()["kernel_launches_per_step"] == 6
    ctx.use_persistent(2)
    ctx.set_tile_variant(3)
    got.append(advance())
    assert ctx.info()["per_class_tiles"] == 0 and ctx.info()["persistent"] == 2
    ctx.use_persistent(1)
    got.append(advance())
    ctx.close()
    for g in got:
        assert all(np.array_equal(a, b) for a, b in zip(g, want))


def test_autotune_tries_the_resident_step_where_it_fits():
    from paper_1901_02955_gb300 import Context
    w = dry(336, 504)
    ctx = Context(w, dtype="f32")
    ctx.set_state(w.Y)
    ctx.step(2)
    want = ctx.get_state()
    ctx.set_state(w.Y)
    ctx.autotune(steps=2)
    ctx.step(2)
    assert np.array_equal(ctx.get_state(), want)
    ctx.close()


@pytest.mark.parametrize("make,dtype,nx,nz,nu,mode", [
    (moist, "f64", 446, 108, 0.0, 0), (moist, "f32", 486, 344, 0.0, 0),
    (moist, "f32", 628, 229, 0.0, 0), (dry, "f32", 768, 256, 0.0, 0),
    (dry, "f32", 1039, 179, 75.0, 0), (dry, "f64", 544, 160, 0.0, 0),
    (dry, "f64", 544, 160, 0.0, 1), (dry, "f64", 282, 427, 75.0, 1),
    (moist, "f64", 346, 162, 0.0, 1)])
def test_heights_do_not_spill_a_few_tiles_into_another_round(make, dtype, nx, nz, nu, mode):
    """The heights keep such grids within the co-resident tiles, or well into the next round: a few
    tiles more than are co-resident cost a whole round (446 x 108 moist FP64: 154 tiles on 152
    places, 1.6 times the step of 126)."""
    import torch
    from paper_1901_02955_gb300 import Context
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("grids chosen for 152 SMs")
    w = make(nx, nz) if make is moist else W.density_current(nx=nx, nz=nz, nu=nu)
    ctx = Context(w, dtype=dtype)
    ctx.use_persistent(mode)
    info = ctx.info()
    ctx.close()
    over = info["tiles_total"] / info["persistent_grid"]  # (that many CTAs, or every tile)
    assert over == 1.0 or over > 1.15, info
