"""Serving from a tight pool: the scratch that only makes a batch faster (the poses in tile order) keeps no other request
out.  A pool with room for two large requests at their least holds both at once."""
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


def _serve_two(mhc, pool_bytes, scenes):
    ctx = mhc.Context(0, 8 << 20)
    srv = mhc.Server(ctx, pool_bytes, large_slots=2, max_batch=1)
    try:
        warm = srv.submit(scenes[0])                               # kernels loaded, pinned buffers allocated
        assert srv.poll(warm, None, timeout_us=60_000_000)
        srv.release(warm)
        srv.pause(True)
        tickets = [srv.submit(sc) for sc in scenes]
        srv.pause(False)
        outs = []
        for t, sc in zip(tickets, scenes):
            out = mhc.alloc_risk(sc, device="cpu")
            assert srv.poll(t, out, timeout_us=60_000_000)
            outs.append(out)
        times = [srv.times(t)[0] for t in tickets]
        for t in tickets:
            srv.release(t)
        return outs, times
    finally:
        srv.stop()
        ctx.close()
        torch.cuda.empty_cache()


def test_two_large_requests_at_their_least(mhc):
    scenes = [S.stress32(4), S.stress32(5)]                       # 507,904 tiles: no block records in their scratch
    lay = mhc.layout(scenes[0])
    resident = lay["run_bytes"] - lay["scratch"] + 256
    extra = _al(512 * 32 * 64 * 50) + _al(128 * 32 * 64) + 256 + _al(128 * 507904)   # poses, order and list
    least = resident + lay["scratch"] - extra
    cs = [mhc.as_c(sc) for sc in scenes]
    tight, times = _serve_two(mhc, 2 * least + (1 << 20), cs)
    assert times[1][1] < times[0][2], times                        # the second was launched while the first ran
    roomy, _ = _serve_two(mhc, 4 * (least + extra), cs)
    for a, b in zip(tight, roomy):
        for k in a:
            if k == "scalars":
                torch.testing.assert_close(a[k], b[k], rtol=1e-12, atol=1e-18)
            else:
                assert torch.equal(a[k], b[k]), k


def test_a_long_queue_does_not_slow_its_requests(mhc):
    """One large slot: nothing in the queue could run beside the batch, so it gets its larger scratch."""
    sc = mhc.as_c(S.stress32(4))
    lay = mhc.layout(sc)
    ctx = mhc.Context(0, 8 << 20)
    srv = mhc.Server(ctx, 3 * lay["run_bytes"], large_slots=1, max_batch=1)

    def spans(n):
        srv.pause(True)
        tickets = [srv.submit(sc) for _ in range(n)]
        srv.pause(False)
        out = []
        for t in tickets:
            assert srv.poll(t, None, timeout_us=60_000_000)
            ns, _ = srv.times(t)
            out.append(ns[2] - ns[1])
            srv.release(t)
        return sorted(out)[n // 2]

    try:
        spans(1)                                                   # kernels loaded, pinned buffers allocated
        alone = spans(1)
        assert spans(6) < 1.5 * alone
    finally:
        srv.stop()
        ctx.close()
        torch.cuda.empty_cache()
