"""Outline pairs in the tile-ordered collision layouts: a first look (rectangles inside the outlines, the two edges that
face each other) decides most candidates, the others take a lane per edge.  Outlines where that can go wrong: three
vertices, sixteen (32 edges a pair), slivers, off-centre ones with the pose point outside (no rectangle inside), mixed with
rectangles and discs, in few blocks, in halved and in many.  The reference is the plainest layout, whose every candidate
takes the whole test: tables bit for bit."""
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


def _ngon(n, rx, ry, x0=0.0, y0=0.0, turn=0.0):
    t = turn + 2.0 * np.pi * np.arange(n) / n
    return np.stack([x0 + rx * np.cos(t), y0 + ry * np.sin(t)], axis=1).astype(np.float32)


OUTLINES = {
    "triangles": [_ngon(3, 3.0, 1.5), _ngon(3, 2.0, 2.0, turn=0.5)],
    "sixteen": [_ngon(16, 2.4, 1.0), _ngon(16, 3.0, 1.3, 0.4, -0.2)],
    "slivers": [_ngon(4, 4.0, 0.05), _ngon(5, 3.0, 0.2, turn=0.3)],
    "off centre": [_ngon(6, 1.5, 0.8, 3.0, 0.5), _ngon(7, 1.0, 1.0, -2.0, 1.5)],
    "mixed": [None, _ngon(9, 2.2, 0.9), None, S.chamfered_outline(4.5, 1.8, 0.35)],
}


@pytest.mark.parametrize("shape", sorted(OUTLINES))
@pytest.mark.parametrize("n_acc,n_str,n_ped", [(3, 2, 3), (21, 21, 7), (33, 41, 9)])
def test_outline_pairs(mhc, shape, n_acc, n_str, n_ped):
    sc = S.intersection11(7, 33, n_acc, n_str, n_ped, n_ped)
    cars = [o for o in sc.objects if o.kind == S.VEHICLE][:4 if n_acc > 30 else 5]
    peds = [o for o in sc.objects if o.kind != S.VEHICLE][:2]
    forms = OUTLINES[shape]
    cars = [dataclasses.replace(o, outline=forms[q % len(forms)]) for q, o in enumerate(cars)]
    sc = dataclasses.replace(sc, objects=cars + peds, ego=0)
    ctx = mhc.Context(0, mhc.layout(sc)["scratch"] + (8 << 20))
    try:
        ctx.set_option(mhc.MHC_OPT_COLLIDE_VARIANT, 1)
        poses = mhc.generate(ctx, sc)
        want = mhc.detect(ctx, sc, poses)
        torch.cuda.synchronize()
        assert int((want >= 0).sum()) > 0
        for variant in (7, 4):
            ctx.set_option(mhc.MHC_OPT_COLLIDE_VARIANT, variant)
            for cull in (1, 0):
                ctx.set_option(mhc.MHC_OPT_CULL, cull)
                got = mhc.detect(ctx, sc, poses)
                torch.cuda.synchronize()
                assert torch.equal(got, want), (variant, cull)
            ctx.set_option(mhc.MHC_OPT_CULL, 1)
    finally:
        ctx.close()
        torch.cuda.empty_cache()
