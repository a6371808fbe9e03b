"""The large-scene collision layout (a warp per listed block of tile-ordered hypotheses) at the sizes where it can go
wrong: strips of the tile order that do not divide the grid, run backwards or along the other axis, ragged tiles, more
than one chunk of 32 steps, eight tiles per listing warp, and an arena without room for the tile-ordered poses.  The
reference is the plainest layout (one CTA per tile, ascending hypotheses, nothing culled), itself checked against the
oracle: tables and fixed-point sums bit for bit, the FP64 totals to the rounding of their order of addition."""
import dataclasses

import numpy as np
import pytest

from paper_2005_06773_gb300 import scenarios as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def mhc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_06773_gb300 import mhc as m
    return m


def _scene(n_a, n_b, n_steps=37, model=S.MODEL_OT):
    """Four cars and two pedestrians; the first car has the n_a x n_b grid, the others other shapes."""
    sc = S.intersection11(21, n_steps, 6, 9, 4, 9)
    objs = [sc.objects[q] for q in (0, 1, 2, 3, 7, 8)]
    ga = S.accel_grid_paper(n_a, -8.0, 3.0) if n_a >= 3 else S.linspace(-3.0, 1.0, n_a)
    objs[0] = dataclasses.replace(objs[0], grid_a=ga, grid_b=S.linspace(-0.3, 0.3, n_b))
    objs[1] = dataclasses.replace(objs[1], grid_a=S.accel_grid_paper(6, -9.7, 9.7), grid_b=S.linspace(-0.05, 0.05, 67))
    return dataclasses.replace(sc, objects=objs, model=model)


def _outputs(mhc, ctx, sc, variant, cull, w):
    ctx.set_option(mhc.MHC_OPT_COLLIDE_VARIANT, variant)
    ctx.set_option(mhc.MHC_OPT_CULL, cull)
    p, t, r = mhc.evaluate(ctx, sc, weights=w)
    d = mhc.detect(ctx, sc, p)
    torch.cuda.synchronize()
    assert torch.equal(t, d)
    return t, r


def _same(a, b):
    assert torch.equal(a[0], b[0])
    for k in a[1]:
        if k == "scalars":
            np.testing.assert_allclose(a[1][k].cpu().numpy(), b[1][k].cpu().numpy(), rtol=1e-12, atol=1e-18)
        else:
            assert torch.equal(a[1][k], b[1][k]), k


@pytest.mark.parametrize("n_a,n_b", [(1, 1), (1, 40), (40, 1), (2, 33), (5, 13), (3, 47), (31, 33), (64, 5)])
@pytest.mark.parametrize("ego", [0, 1, 4])
def test_tile_order_and_ragged_tiles(mhc, n_a, n_b, ego):
    sc = dataclasses.replace(_scene(n_a, n_b), ego=ego)
    w = S.random_weights(sc, 3)
    ctx = mhc.Context(0, 128 << 20)
    try:
        ref = _outputs(mhc, ctx, sc, 1, 0, w)
        assert int((ref[0] >= 0).sum()) > 0
        for cull in (1, 0):
            _same(_outputs(mhc, ctx, sc, 4, cull, w), ref)
    finally:
        ctx.close()


def test_eight_tiles_per_listing_warp_and_small_arena(mhc):
    """About 64,000 tiles of 8 cars; the same with an arena that holds neither the tile-ordered poses nor the list."""
    sc = S.stress32(5, 8, 64, 48, 33)
    lay = mhc.layout(sc)
    n_tiles = 28 * 48 * 48
    tables = []
    for arena in (lay["scratch"], lay["scratch"] - 128 * 4 * n_tiles + (4 << 20)):
        ctx = mhc.Context(0, arena)
        try:
            ctx.set_option(mhc.MHC_OPT_COLLIDE_VARIANT, 4)
            _, t, r = mhc.evaluate(ctx, sc)
            torch.cuda.synchronize()
            tables.append((t, r))
        finally:
            ctx.close()
    ctx = mhc.Context(0, lay["scratch"])
    try:
        ctx.set_option(mhc.MHC_OPT_COLLIDE_VARIANT, 5)
        _, t, r = mhc.evaluate(ctx, sc)
        torch.cuda.synchronize()
        for got in tables:
            _same(got, (t, r))
        assert int((t >= 0).sum()) > 0
    finally:
        ctx.close()
        torch.cuda.empty_cache()
