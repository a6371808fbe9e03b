"""A submitted request owns its scenario: what the caller does to its arrays afterwards (outlines, lane paths, grids,
parameters, weights) changes no result, also where requests share a batch and are laid out once more for it."""
import dataclasses

import numpy as np
import pytest

from paper_2005_06773_gb300 import scenarios as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_arrays_overwritten_after_submission():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_06773_gb300 import mhc
    scenes = [S.with_outlines(S.intersection11(31, 20, 5, 7, 3, 3), cut=0.35),
              S.with_lane_paths(S.intersection11(32, 22, 5, 7, 3, 3)), S.with_outlines(S.intersection11(33, 18, 7, 5, 3, 3))]
    scenes = [dataclasses.replace(sc, objects=[dataclasses.replace(o, params=S.DEFAULT_VEH_PARAMS * np.float32(1.1))
                                               if o.kind == S.VEHICLE else o for o in sc.objects]) for sc in scenes]
    weights = [S.random_weights(sc, 40 + q) for q, sc in enumerate(scenes)]
    solo = mhc.Context(0, 256 << 20)
    refs = [{k: v.clone() for k, v in mhc.run(solo, sc, weights=w).items()} for sc, w in zip(scenes, weights)]
    solo.close()
    ctx = mhc.Context(0, 64 << 20)
    srv = mhc.Server(ctx, 1 << 30)
    try:
        srv.pause(True)
        tickets = []
        for sc, w in zip(scenes, weights):
            mine = mhc.as_c(dataclasses.replace(sc, objects=[dataclasses.replace(
                o, **{f: np.array(getattr(o, f)) for f in ("grid_a", "grid_b", "params", "outline", "paths")
                      if getattr(o, f) is not None}) for o in sc.objects]))
            w = [np.array(v) for v in w]
            tickets.append((srv.submit(mine, w), mine))
            for a in mine._keep + w:
                a[...] = np.nan
        srv.pause(False)
        for (t, mine), sc, ref in zip(tickets, scenes, refs):
            out = mhc.alloc_risk(sc, device="cpu")
            assert srv.poll(t, out, timeout_us=10_000_000)
            assert srv.times(t)[1] == len(scenes)          # one batch
            for k in out:
                if k == "scalars":
                    np.testing.assert_allclose(out[k].numpy(), ref[k].numpy(), rtol=1e-12, atol=1e-18)
                else:
                    np.testing.assert_array_equal(out[k].numpy(), ref[k].numpy(), err_msg=k)
            srv.release(t)
    finally:
        srv.stop()
        ctx.close()
