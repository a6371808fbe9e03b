"""Path hypotheses of vehicles whose wheelbase is far from a car's: the parameters are only required to be positive and
finite.  In the kinematic model such a long wheelbase (in the first case the sum of the lever arms overflows) does not turn
the vehicle, and every pose is a number."""
import dataclasses
import math

import numpy as np
import pytest

from paper_2005_06773_gb300 import scenarios as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("lever", [3e38, 1e30, 1e13])
def test_wide(lever):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_06773_gb300 import mhc
    sc = S.with_lane_paths(S.intersection11(11, 20, 5, 7, 3, 3))
    car = next(o for o in sc.objects if o.paths is not None)
    p = np.array(S.DEFAULT_VEH_PARAMS, np.float32)
    p[2] = p[3] = lever
    sc = dataclasses.replace(sc, objects=[dataclasses.replace(car, params=p), sc.objects[-1]], ego=0, model=S.MODEL_KIN)
    ctx = mhc.Context(0, 16 << 20)
    try:
        pose = {k: v.cpu().numpy()[: car.n_hyp * sc.n_steps] for k, v in mhc.generate(ctx, sc).items()}
    finally:
        ctx.close()
    for k, v in pose.items():
        assert np.isfinite(v).all(), k
    np.testing.assert_allclose(pose["c"], math.cos(car.psi0), atol=1e-6)
    np.testing.assert_allclose(pose["s"], math.sin(car.psi0), atol=1e-6)
