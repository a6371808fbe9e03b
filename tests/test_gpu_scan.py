"""The risk scan of a finished table in its two forms (small tables; large ones with histograms in shared memory) where it
can go wrong: ragged rows and columns, the EGO object first or second of its pairs or in few of them, hits crowded into
few steps or spread over many, horizons at the histograms' limits, entries that are no step of the horizon.  The fused
evaluation accumulates the same fixed-point terms at the collisions themselves: integers and fixed-point sums are equal
bit for bit, FP64 sums to the rounding of their order of addition."""
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


def _same(got, want):
    for k in want:
        if k in ("scalars", "naive", "cond", "indep"):
            np.testing.assert_allclose(got[k].cpu().numpy(), want[k].cpu().numpy(), rtol=1e-12, atol=1e-18)
        else:
            assert torch.equal(got[k], want[k]), k


def _scene(n_obj, n_a, n_b, n_steps, crowded):
    sc = S.stress32(5, 8, n_a, n_b, n_steps)
    objs = list(sc.objects)[:n_obj]
    if crowded:
        objs = [dataclasses.replace(o, x0=3.0 * q, y0=0.2 * q, psi0=0.1 * q) for q, o in enumerate(objs)]
    return dataclasses.replace(sc, objects=objs)


@pytest.mark.parametrize("n_obj,n_a,n_b,n_steps", [(2, 3, 1, 5), (3, 13, 5, 31), (4, 21, 23, 1100), (8, 27, 32, 33),
                                                   (8, 29, 30, 1024), (8, 29, 30, 1025)])
@pytest.mark.parametrize("ego", [0, 1])
@pytest.mark.parametrize("crowded", [False, True])
def test_scan_equals_fused(mhc, n_obj, n_a, n_b, n_steps, ego, crowded):
    sc = dataclasses.replace(_scene(n_obj, n_a, n_b, n_steps, crowded), ego=ego)
    w = S.random_weights(sc, 3)
    ctx = mhc.Context(0, mhc.layout(sc)["scratch"] + (8 << 20))
    try:
        _, table, want = mhc.evaluate(ctx, sc, weights=w)
        _same(mhc.assess(ctx, sc, table, weights=w), want)
        assert not crowded or int(want["count"].sum()) > 0
        torch.cuda.synchronize()
    finally:
        ctx.close()
        torch.cuda.empty_cache()


def test_entries_outside_the_horizon_do_not_count(mhc):
    sc = _scene(3, 13, 5, 31, True)
    ctx = mhc.Context(0, 64 << 20)
    try:
        _, table, want = mhc.evaluate(ctx, sc)
        spoiled = table.clone()
        spoiled[(table < 0).nonzero()[::2]] = 31
        spoiled[(table < 0).nonzero()[1::2]] = -7
        _same(mhc.assess(ctx, sc, spoiled), want)
        torch.cuda.synchronize()
    finally:
        ctx.close()
