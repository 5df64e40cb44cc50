"""The 3-D stage as a march along z (the first tile shape of the inviscid 3-D families) against the
one-shot tiles, on grids at the edges of its tiles: fewer columns than a warp or a tile, one more
than a tile, the fewest levels, ragged level counts, every launch mode, periodic and walled sides,
slabs. The dry step agrees bitwise (the same per-cell and per-face arithmetic); with the saturation
adjustment within 1e-6 of each field's largest magnitude, a few units in the last place, as for
the other tile shapes. The temperature inversion of the FP32 kernels (pairs of floats) is checked
through the adjustment itself: an FP32 context's result against an FP64 context's on the same
FP32 state."""
import dataclasses

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


def advance(w, dtype, variant, mode, steps=2):
    from paper_1901_02955_gb300 import Context
    ctx = Context(w, dtype=dtype)
    ctx.set_tile_variant(variant)
    info = ctx.info()
    try:
        ctx.use_persistent(mode)
    except Exception:
        assert mode == 2  # more tiles than can be resident at once
        ctx.close()
        return None, info
    ctx.set_state(w.Y)
    ctx.step(steps)
    out = ctx.get_state()
    ctx.close()
    return out, info


WALLS = (W.REFLECT,) * 6


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("n", [(3, 3, 3), (31, 8, 5), (32, 9, 4), (33, 7, 37), (64, 17, 67), (5, 40, 12)])
@pytest.mark.parametrize("walls", [False, True])
def test_dry_march_equals_tiles_bitwise(n, dtype, walls):
    w = W.add_random_motion(W.dry_bubble_3d(nx=n[0], ny=n[1], nz=n[2]))
    if walls:
        w = dataclasses.replace(w, bc=(W.REFLECT, W.REFLECT, W.NOSLIP, W.NOSLIP) + w.bc[4:])
    ref, info = advance(w, dtype, 1, 0)
    assert info["tile"] == (8, 8, 4)
    for mode in (0, 1, 2):
        out, info = advance(w, dtype, 0, mode)
        assert info["tile"][:2] == (32, 8)
        if out is not None:
            assert np.array_equal(out, ref), mode


@pytest.mark.parametrize("n", [(3, 3, 18), (33, 9, 20), (40, 17, 39)])
@pytest.mark.parametrize("full", [False, True])
def test_moist_march_agrees_with_tiles(n, full):
    make = W.jovian_rce if full else W.jovian
    w = W.add_random_motion(make(nx=n[0], ny=n[1], nz=n[2], Lx=390.0 * n[0], Ly=390.0 * n[1]))
    tiles = 1 if full else 2  # the one-shot shape follows the marching ones
    ref, info = advance(w, "f32", tiles, 0)
    assert info["tile"] == (8, 8, 4)
    scale = np.abs(ref).reshape(w.nv, -1).max(axis=1)
    for v in range(tiles):
        for mode in (0, 1, 2):
            out, info = advance(w, "f32", v, mode)
            assert info["tile"][0] == 32
            if out is None:
                continue
            d = np.abs(out - ref).reshape(w.nv, -1).max(axis=1)
            assert np.all(d <= 1e-6 * np.maximum(scale, 1e-30)), (v, mode, d / scale)


def test_march_over_linked_slabs_equals_the_whole_domain():
    from paper_1901_02955_gb300 import Context
    w = W.add_random_motion(W.dry_bubble_3d(nx=75, ny=20, nz=24))
    ref, _ = advance(w, "f32", 0, 0)
    HALO = 3
    cuts = [0, 34, 75]
    parts = [dataclasses.replace(w, nx=b - a, Y=np.ascontiguousarray(w.Y[..., a:b]),
                                 bc=(HALO, HALO) + w.bc[2:]) for a, b in zip(cuts, cuts[1:])]
    ctx = Context(parts, dtype="f32")
    ctx.set_tile_variant(0)
    for d in range(2):
        ctx.link_halo(d, 0, 1 - d)
        ctx.link_halo(d, 1, 1 - d)
    for d, p in enumerate(parts):
        ctx.set_state(p.Y, domain=d)
    ctx.step(2)
    out = np.concatenate([ctx.get_state(domain=d) for d in range(2)], axis=3)
    ctx.close()
    assert np.array_equal(out, ref)


def test_adjustment_in_pairs_of_floats_tracks_fp64():
    """Saturated and subsaturated Jovian cells: the FP32 context's adjusted state against the FP64
    context's on the same FP32 values. The adjusted vapour follows its saturation pressure, which
    FP32 holds to (|a| + 2) 2^-24 with |a| < 26 the exponent (the adjustment's own stop test
    allows four times that): 4 * 28 * 2^-24 = 6.7e-6 of the species' largest density."""
    from paper_1901_02955_gb300 import Context
    w = W.jovian(nx=16, ny=16, nz=64, noise_K=2.0)
    Y = w.Y.astype(np.float32)
    Y[-1] *= np.float32(0.99)  # about 1 % colder than the saturation the vapours are capped at
    out = {}
    for dtype in ("f32", "f64"):
        ctx = Context(w, dtype=dtype)
        ctx.set_state(Y.astype(np.float64))
        ctx.saturation_adjust()
        out[dtype] = ctx.get_state()
        ctx.close()
    moved = np.abs(out["f64"] - Y.astype(np.float64)).reshape(w.nv, -1).max(axis=1)
    assert moved[1] > 1e-4  # water condenses (the column stays too warm for ammonia ice)
    for f in range(1, 1 + w.nvapor * (1 + w.ncond)):
        i = f - 1 if f <= w.nvapor else (f - 1 - w.nvapor) // w.ncond
        scale = np.abs(Y[1 + i]).reshape(w.nz, -1).max(axis=1)[:, None, None]
        d = np.abs(out["f32"][f] - out["f64"][f])
        assert np.all(d <= 6.7e-6 * scale), (f, (d / scale).max())
