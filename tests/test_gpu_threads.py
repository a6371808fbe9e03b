"""Several host threads, each with a context of its own: calls whose kernels opt in to different amounts of dynamic shared
memory run side by side, and none of them fails or changes its results."""
import dataclasses
import threading
import time

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


def _together(calls, seconds=4.0):
    """Every call in a thread of its own, again and again until one fails or the time is over."""
    errors, stop, end = [], threading.Event(), time.time() + seconds

    def work(call):
        try:
            while not stop.is_set() and time.time() < end:
                call()
        except Exception as e:
            errors.append(e)
            stop.set()

    threads = [threading.Thread(target=work, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors


def test_assess_horizons(mhc):
    """Scans with histograms (from 4,864 tiles) of 1,024 and 800 steps."""
    one = S.tiny_crossing(1).objects[0]
    one = dataclasses.replace(one, grid_a=one.grid_a[:1], grid_b=one.grid_b[:1])
    ctxs, calls = [], []
    for n in (1024, 800) * 4:
        sc = mhc.as_c(dataclasses.replace(S.tiny_crossing(1), objects=[one] * 101, n_steps=n))
        ctx, st = mhc.Context(0, 256 << 20), torch.cuda.Stream()
        table = torch.full((mhc.layout(sc)["n_entries"],), 7, dtype=torch.int16, device="cuda")
        out = mhc.alloc_risk(sc)
        torch.cuda.synchronize()
        ctxs.append((ctx, out))
        calls.append(lambda ctx=ctx, sc=sc, table=table, out=out, st=st: mhc.assess(ctx, sc, table, None, out, stream=st))
    try:
        _together(calls)
        for _, out in ctxs:
            assert int(out["count"].sum()) == 101 * 100 // 2
    finally:
        for ctx, _ in ctxs:
            ctx.close()


@pytest.mark.parametrize("variant", [1, 3])
def test_evaluate_horizons(mhc, variant):
    """Collision layouts with a CTA per tile, 160 and 60 steps."""
    ctxs, calls, refs = [], [], {}
    for n in (160, 60) * 4:
        sc = mhc.as_c(dataclasses.replace(S.tiny_crossing(3, start=18.0), n_steps=n))
        ctx, st = mhc.Context(0, 32 << 20), torch.cuda.Stream()
        ctx.set_option(mhc.MHC_OPT_COLLIDE_VARIANT, variant)
        bufs = mhc.evaluate(ctx, sc)
        torch.cuda.synchronize()
        refs.setdefault(n, bufs[1].clone())
        ctxs.append((ctx, n, bufs))
        calls.append(lambda ctx=ctx, sc=sc, b=bufs, st=st: mhc.evaluate(ctx, sc, b[0], b[1], None, b[2], stream=st))
    try:
        _together(calls, 2.0)
        for _, n, bufs in ctxs:
            assert torch.equal(bufs[1], refs[n])
    finally:
        for ctx, _, _ in ctxs:
            ctx.close()
