"""The small-scene collision layout (a CTA per active block) at the sizes where it can go wrong: few blocks, each with a
CTA of its own, and many, listed; ragged tiles, more than one chunk of 32 steps, batches that end a chunk, the EGO
object on either side of a pair or in none, first hits spread over many steps or crowded into few (the two ways their
risk terms are summed), outlines, no room for the list.  The reference is the plainest layout (one CTA per tile,
nothing culled), itself checked against the oracle: tables and fixed-point sums bit for bit, the FP64 totals to the
rounding of their order of addition."""
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


def _scene(n_obj, n_a, n_b, n_steps, crowded):
    """n_obj cars of n_a x n_b hypotheses; crowded: side by side, so that hits come within a few steps."""
    sc = S.stress32(5, 8, max(n_a, 3), n_b, n_steps)
    objs = list(sc.objects)[:n_obj]
    if crowded:
        objs = [dataclasses.replace(o, x0=3.0 * q, y0=0.2 * q, psi0=0.1 * q) for q, o in enumerate(objs)]
    if n_a < 3:
        objs = [dataclasses.replace(o, grid_a=S.linspace(-3.0, 1.0, n_a)) for o in objs]
    return dataclasses.replace(sc, objects=objs)


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
        if k in ("scalars", "naive", "cond", "indep"):
            np.testing.assert_allclose(a[1][k].cpu().numpy(), b[1][k].cpu().numpy(), rtol=1e-12, atol=1e-18)
        else:
            assert torch.equal(a[1][k], b[1][k]), k


@pytest.mark.parametrize("n_obj,n_a,n_b,n_steps", [(2, 1, 1, 40), (3, 5, 13, 31), (3, 33, 2, 97), (4, 31, 33, 37), (5, 23, 29, 64),
                                                   (4, 31, 33, 9), (4, 19, 17, 70)])
@pytest.mark.parametrize("ego", [0, 1])
@pytest.mark.parametrize("crowded", [False, True])
def test_blocks(mhc, n_obj, n_a, n_b, n_steps, ego, crowded):
    sc = dataclasses.replace(_scene(n_obj, n_a, n_b, n_steps, crowded), ego=ego)
    if n_obj == 3:
        sc = S.with_outlines(sc, 0.35)
    w = S.random_weights(sc, 3)
    ctx = mhc.Context(0, 256 << 20)
    try:
        ref = _outputs(mhc, ctx, sc, 1, 0, w)
        assert not crowded or int((ref[0] >= 0).sum()) > 0
        for cull in (1, 0):
            _same(_outputs(mhc, ctx, sc, 7, cull, w), ref)
    finally:
        ctx.close()


def test_small_arena(mhc):
    """An arena that holds neither the tile-ordered poses nor the list."""
    sc = S.intersection11(5)
    lay = mhc.layout(sc)
    n64 = [(o.n_hyp + 63) // 64 for o in sc.objects]
    blocks = 4 * sum(a * b for i, a in enumerate(n64) for b in n64[i + 1:])
    outs = []
    for arena in (lay["scratch"], lay["scratch"] - 32 * blocks + (64 << 10)):
        ctx = mhc.Context(0, arena)
        try:
            ctx.set_option(mhc.MHC_OPT_COLLIDE_VARIANT, 7)
            _, t, r = mhc.evaluate(ctx, sc)
            torch.cuda.synchronize()
            outs.append((t, r))
        finally:
            ctx.close()
    _same(outs[1], outs[0])
