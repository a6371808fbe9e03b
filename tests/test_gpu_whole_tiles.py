"""The large-scene collision layout without its list (culling off, or an arena without room for the poses in tile order):
from 64 tiles per SM a warp walks a whole 64 x 64 tile of ascending hypotheses.  The reference is the layout with a warp
per quarter tile: tables and fixed-point sums bit for bit, the FP64 totals to the rounding of their order of addition."""
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


def _same(a, b):
    assert torch.equal(a[1], b[1])
    for k in a[2]:
        if k in ("scalars", "naive", "cond", "indep"):
            np.testing.assert_allclose(a[2][k].cpu().numpy(), b[2][k].cpu().numpy(), rtol=1e-12, atol=1e-18)
        else:
            assert torch.equal(a[2][k], b[2][k]), k


@pytest.mark.parametrize("n_obj,n_a,n_b,n_steps", [(12, 41, 21, 33), (12, 33, 25, 64), (12, 29, 31, 5), (160, 3, 1, 35)])
@pytest.mark.parametrize("ego", [0, 2])
def test_without_culling(mhc, n_obj, n_a, n_b, n_steps, ego):
    """Ragged tiles of 861, 825 and 899 hypotheses a side (12,936 tiles; 12,870 tiles of 3 x 3 hypotheses)."""
    sc = S.stress32(7, 12, n_a, n_b, n_steps)
    objs = [dataclasses.replace(o, x0=o.x0 + q // 12) for q, o in enumerate((sc.objects * 14)[:n_obj])]
    sc = dataclasses.replace(sc, objects=objs, ego=ego)
    w = S.random_weights(sc, 3)
    ctx = mhc.Context(0, mhc.layout(sc)["scratch"])
    try:
        ctx.set_option(mhc.MHC_OPT_CULL, 0)
        outs = []
        for variant in (5, 4):
            ctx.set_option(mhc.MHC_OPT_COLLIDE_VARIANT, variant)
            outs.append(mhc.evaluate(ctx, sc, weights=w))
            torch.cuda.synchronize()
            assert torch.equal(outs[-1][1], mhc.detect(ctx, sc, outs[-1][0]))
        _same(outs[1], outs[0])
        assert n_steps < 10 or int((outs[0][1] >= 0).sum()) > 0    # (five steps: nobody meets yet)
    finally:
        ctx.close()


def test_time_without_culling(mhc):
    """12 cars of 1,100 hypotheses: the sweep of whole tiles takes two thirds of the quarter tiles' time (both measured
    here; with a walk over every 32 x 32 block it took 1.07 times as long)."""
    sc = mhc.as_c(S.stress32(7, 12, 50, 22, 30))
    ctx = mhc.Context(0, mhc.layout(sc)["scratch"])
    best = {}
    try:
        ctx.set_option(mhc.MHC_OPT_CULL, 0)
        poses = mhc.generate(ctx, sc)
        table = mhc.detect(ctx, sc, poses)
        ctx.profile(True)
        for variant in (5, 4) * 6:
            ctx.set_option(mhc.MHC_OPT_COLLIDE_VARIANT, variant)
            ctx.profile_read(reset=True)
            mhc.detect(ctx, sc, poses, table)
            torch.cuda.synchronize()
            best[variant] = min(best.get(variant, 1e9), ctx.profile_read(reset=True)["collide"][0])
    finally:
        ctx.close()
    assert best[4] < 0.85 * best[5], best
