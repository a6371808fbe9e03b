"""The default collision layout goes by the number of tiles alone: scenes of one structure take the same kernels whatever
their horizon, grid values and speeds (a replayed plan keeps the kernels of the scene it was created with)."""
import dataclasses

import pytest

from paper_2005_06773_gb300 import scenarios as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("make", [lambda n: S.intersection11(3, n), lambda n: S.stress32(3, 16, 8, 28, n)])
def test_same_kernels(make):
    """1,445 and 1,920 tiles: a listing and the kernel of layout 7."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_06773_gb300 import mhc
    for n_steps in (15, 60):
        for v0 in (1.0, 12.0, 30.0):
            sc = make(n_steps)
            sc = dataclasses.replace(sc, objects=[dataclasses.replace(o, v0=v0) if o.kind == S.VEHICLE else o for o in sc.objects])
            ctx = mhc.Context(0, max(1 << 20, mhc.layout(sc)["scratch"]))
            try:
                ctx.profile(True)
                mhc.evaluate(ctx, sc)
                torch.cuda.synchronize()
                assert ctx.profile_read()["collide"][1] == 2, (n_steps, v0)
            finally:
                ctx.close()
