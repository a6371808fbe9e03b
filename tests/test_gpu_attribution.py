"""The EGO walk's attribution per object and step in its two forms: with atomics (few cells) and summed by a kernel of
its own from the terms left in the cells (2^19 cells and more).  The sums are fixed point, so a batch that takes the
second form gives, scenario by scenario, the first form's outputs bit for bit; a scene that takes the second form on
its own is held to the identity sum_h p_h P_cond(h) = sum over objects = sum over steps, each term rounded to 2^-40."""
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


def _cells(sc):
    return sc.objects[sc.ego].n_hyp * sc.n_steps * len(sc.objects)


@pytest.mark.parametrize("shapes", [
    [(21, 21, 30), (3, 5, 7)] * 4,                     # one window of cells, a ragged last group of hypotheses
    [(4, 4, 230), (3, 2, 1), (17, 2, 190)] * 8,        # several windows, which cut a step
])
def test_batch_equals_its_scenarios(mhc, shapes):
    scs = [S.intersection11(5 + q, n, a, b, 5, 5) for q, (a, b, n) in enumerate(shapes)]
    assert sum(map(_cells, scs)) >= 1 << 19 > max(map(_cells, scs))
    ctx = mhc.Context(0, 512 << 20)
    _, _, both = mhc.evaluate_batch(ctx, scs)
    ones = [mhc.evaluate(ctx, sc)[2] for sc in scs]
    torch.cuda.synchronize()
    for k in both:
        want = torch.cat([one[k].flatten() for one in ones]).cpu().numpy()
        got = both[k].flatten().cpu().numpy()
        if k == "scalars":
            np.testing.assert_allclose(got, want, rtol=1e-12, atol=1e-18)
        else:
            assert np.array_equal(got, want), k


@pytest.mark.parametrize("n_a,n_b,n_steps", [(64, 32, 50), (23, 21, 333)])
def test_one_scene(mhc, n_a, n_b, n_steps):
    sc = S.intersection11(9, n_steps, n_a, n_b, 3, 3)
    assert _cells(sc) >= 1 << 19
    ctx = mhc.Context(0, 512 << 20)
    _, _, r = mhc.evaluate(ctx, sc, weights=S.random_weights(sc, 4))
    torch.cuda.synchronize()
    total = float(r["scalars"].flatten()[1])
    tol = _cells(sc) * 2.0 ** -40 + 1e-6 * total       # rounding to fixed point; p_h in FP32 against FP64
    assert total > 0.0
    assert abs(float(r["attr_obj"].sum()) - total) <= tol
    assert abs(float(r["attr_step"].sum()) - total) <= tol
