"""Arenas between the least a call runs in and what its fastest kernels want: without room for the poses in tile order, for
the order, or for the list of blocks, layouts 4 and 7 take the kernels of ascending tiles (one launch instead of the
listing and its kernel) with the same results.  The least is searched for, so that the fallback is sure to run."""
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


def _al(n):
    return (n + 255) // 256 * 256


def _evaluate(mhc, sc, variant, arena):
    """(poses, table, outputs, collision launches), or None where the arena is too small."""
    ctx = mhc.Context(0, arena)
    try:
        ctx.set_option(mhc.MHC_OPT_COLLIDE_VARIANT, variant)
        ctx.profile(True)
        p, t, r = mhc.evaluate(ctx, sc, weights=S.random_weights(sc, 3))
        torch.cuda.synchronize()
        return p, t, r, ctx.profile_read()["collide"][1]
    except mhc.MhcError as e:
        assert "NOMEM" in str(e), e
        return None
    finally:
        ctx.close()


@pytest.mark.parametrize("variant", [4, 7])
@pytest.mark.parametrize("outlines", [False, True])
def test_every_step_of_room(mhc, variant, outlines):
    sc = S.intersection11(5, 40, 21, 23)
    if outlines:
        sc = S.with_outlines(sc, 0.35)
    n32 = [-(-o.n_hyp // 32) for o in sc.objects]
    n64 = [-(-o.n_hyp // 64) for o in sc.objects]
    tiles = sum(n64[a] * n64[b] for a, b in sc.pairs())
    poses, order, lists = _al(512 * sum(n32) * sc.n_steps), _al(128 * sum(n32)), _al(128 * tiles)
    lo, hi = 4096, mhc.layout(sc)["scratch"] // 256           # in 256 bytes: too small, enough
    assert _evaluate(mhc, sc, variant, 256 * lo) is None
    while hi - lo > 1:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if _evaluate(mhc, sc, variant, 256 * mid) else (mid, hi)
    least = 256 * hi
    want = _evaluate(mhc, sc, variant, least + poses + order + 256 + lists)
    assert want[3] == 2 and int((want[1] >= 0).sum()) > 0
    for room in (0, poses, poses + order, poses + order + 256, poses + order + 256 + lists - 256):
        got = _evaluate(mhc, sc, variant, least + room)
        assert got[3] == 1, room
        assert torch.equal(got[1], want[1]), room
        for k in got[2]:
            if k in ("scalars", "naive", "cond", "indep"):
                np.testing.assert_allclose(got[2][k].cpu().numpy(), want[2][k].cpu().numpy(), rtol=1e-12, atol=1e-18)
            else:
                assert torch.equal(got[2][k], want[2][k]), (room, k)
