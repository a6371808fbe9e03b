"""Generation of path hypotheses: the warp takes a short body for the sub-steps in which none of its hypotheses is in the
low-speed regime, and stops early when all have stopped.  A hypothesis's poses must not depend on what shares its warp:
a mixed grid of accelerations (standing start, stop early, late or never) gives, bit for bit, the poses of each
acceleration alone."""
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


@pytest.mark.parametrize("v0", [0.0, 0.4, 6.0, 35.0])
@pytest.mark.parametrize("paths", [1, 3, 7])
@pytest.mark.parametrize("n_steps,substeps", [(1, 1), (37, 4)])
def test_independent_of_the_warp(mhc, v0, paths, n_steps, substeps):
    base = S.with_lane_paths(S.intersection11(11, n_steps, 5, paths, 3, 3))
    car = next(o for o in base.objects if o.paths is not None)
    acc = np.array([3.0, -9.0, 0.0, -0.5, -30.0, 1.0, -4.0, -2.0, 0.0, -6.0, 0.25], dtype=np.float32)
    n_path = car.n_hyp // len(car.grid_a)

    def poses(grid):
        o = dataclasses.replace(car, v0=v0, grid_a=grid)
        sc = dataclasses.replace(base, objects=[o, base.objects[-1]], ego=0, substeps=substeps)
        ctx = mhc.Context(0, 16 << 20)
        try:
            p = mhc.generate(ctx, sc)
            torch.cuda.synchronize()
            n = len(grid) * n_path
            return {k: v.cpu().numpy()[: n * n_steps].reshape(n_steps, n) for k, v in p.items()}
        finally:
            ctx.close()

    mixed = poses(acc)
    for q in range(len(acc)):
        alone = poses(acc[q:q + 1])
        for k in mixed:
            assert np.array_equal(mixed[k][:, q * n_path:(q + 1) * n_path], alone[k]), (k, acc[q])
