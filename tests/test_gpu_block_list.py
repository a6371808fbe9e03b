"""The list of active blocks where poses overflow: a pedestrian of 3e38 m/s leaves FP32 within the horizon, and a tile of
such hypotheses, headings all around, has a box from minus to plus infinity, which meets everything.  Only blocks of the
objects' own tiles may be listed (each object's last 64-wide tile has one 32-wide tile here), and the pairs of objects
whose poses are finite keep the table of the plainest layout."""
import dataclasses
import math

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


@pytest.mark.parametrize("variant", [4, 7])
def test_boxes_without_bounds(mhc, variant):
    sc = S.intersection11(21, 20, 5, 13, 4, 8)
    objs = [dataclasses.replace(o, grid_a=np.linspace(2.5e38, 3.3e38, 4), grid_b=S.linspace(-math.pi, 0.75 * math.pi, 8))
            if o.kind == S.PEDESTRIAN else o for o in sc.objects]
    sc = dataclasses.replace(sc, objects=objs)
    ctx = mhc.Context(0, 64 << 20)
    try:
        ctx.set_option(mhc.MHC_OPT_COLLIDE_VARIANT, 1)
        ctx.set_option(mhc.MHC_OPT_CULL, 0)
        poses = mhc.generate(ctx, sc)
        ref = mhc.detect(ctx, sc, poses)
        ctx.set_option(mhc.MHC_OPT_COLLIDE_VARIANT, variant)
        ctx.set_option(mhc.MHC_OPT_CULL, 1)
        ctx.work(reset=True)
        table = mhc.detect(ctx, sc, poses)
        done = ctx.work()["executed"]
    finally:
        ctx.close()
    assert not bool(torch.isfinite(poses["x"]).all())
    tiles = [-(-o.n_hyp // 32) for o in sc.objects]
    blocks = sum(tiles[a] * tiles[b] for a, b in sc.pairs())
    assert 0 < done <= blocks * sc.n_steps * 1024
    a, b, off = mhc.pair_table(sc)
    finite = 0
    for p in range(len(a)):
        got, want = table[int(off[p]):int(off[p + 1])], ref[int(off[p]):int(off[p + 1])]
        assert int(got.min()) >= -1 and int(got.max()) < sc.n_steps
        if all(objs[int(q)].kind == S.VEHICLE for q in (a[p], b[p])):
            finite += int((want >= 0).sum())
            assert torch.equal(got, want), p
    assert finite > 0
