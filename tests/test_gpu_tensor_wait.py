"""Bounded waits that run out.  Tensor mode with a wait limit of zero: the CTAs give up at their first wait
that is not over at once (many of the larger sizes', not every time: the hardware's own wait takes a
while), let what they have in flight finish, and the next synchronising call reports HOT_ETIMEOUT --
or every wait was over in time and the results are the bits of a call with a limit.  With a limit again,
the context computes what a new one does.  A wait that runs out after an earlier look at the error
flag (a row-band sequence, a replayed capture) is reported all the same."""
import numpy as np
import pytest

from paper_0907_4027_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hot():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0907_4027_gb300 import _build
    _build.build()
    from paper_0907_4027_gb300 import hot as h
    return h


@pytest.mark.parametrize("W,H,M", [(96, 70, 12), (640, 300, 200), (1024, 512, 1000)])
def test_timeout_is_reported_and_recovered_from(hot, W, H, M):
    w = wl.random_case(W, H, M, seed=W, precision="tensor")
    with hot.Hologram.from_workload(w) as h:
        h.gsw(3)
        ref = (h.phase("f32"), *h.fields())
    with hot.Hologram.from_workload(w) as h:
        h.use_graphs(False)
        h.set_wait_limit(0.0)
        h.gsw(3, metrics=False)
        try:
            h.sync()
        except hot.HotError as e:
            assert e.status == hot.HOT_ETIMEOUT
        else:
            assert all(np.array_equal(a, b) for a, b in zip((h.phase("f32"), *h.fields()), ref))
        h.set_wait_limit(2.0)
        h.set_phase(w.phi0)
        h.set_weights(np.ones(M))
        h.gsw(3)
        assert all(np.array_equal(a, b) for a, b in zip((h.phase("f32"), *h.fields()), ref))


@pytest.mark.parametrize("read", ["fields", "metrics", "sharded_end"])
def test_row_band_timeout_after_an_earlier_check(hot, read):
    w = wl.random_case(1024, 1024, 1000, seed=2, precision="tensor")

    def run(limit):
        with hot.Hologram(w.W, 512, w.pitch, w.wavelength, w.focal, precision="tensor") as h:
            h.set_band(w.H, 0)
            h.set_traps(w.xyz)
            h.set_phase(w.phi0[:512 * w.W])
            h.sharded_begin()
            h.sync()
            h.set_wait_limit(limit)
            for k in range(1, 5):
                h.sharded_step(k)
            if read == "sharded_end":
                return np.array(h.sharded_end(4))
            hot._ok(hot.lib.hot_sharded_end(hot._vp(h.ctx), 4, None, None), "hot_sharded_end")
            return np.array(h.fields()[0] if read == "fields" else h.metrics())

    ref = run(2.0)
    try:
        got = run(0.0)
    except hot.HotError as e:
        assert e.status == hot.HOT_ETIMEOUT
    else:
        assert np.array_equal(got, ref)


@pytest.mark.parametrize("read", ["fields", "metrics"])
def test_replayed_capture_timeout(hot, read):
    import torch
    w = wl.random_case(128, 64, 9, seed=6, precision="fast")
    st = torch.cuda.Stream()
    with torch.cuda.stream(st), hot.Hologram.from_workload(w, st.cuda_stream) as h:
        h.use_persistent(True)
        h.gsw(1)
        h.set_wait_limit(0.0)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            h.gsw(5, metrics=False)
        h.sync()
        g.replay()
        with pytest.raises(hot.HotError, match="HOT_ETIMEOUT"):
            getattr(h, read)()


@pytest.mark.parametrize("batch", [False, True])
def test_a_new_limit_reaches_calls_that_were_captured_before(hot, batch):
    """Among 50 runs of a graph's sequence with a limit of zero at least one wait runs out (each has some
    thousand waits for copies from memory)."""
    w = wl.random_case(1024, 1024, 1000, seed=3, precision="tensor")
    with hot.Hologram.from_workload(w) as h, hot.Batch([h]) as b:
        run = (lambda: b.gsw(2)) if batch else (lambda: h.gsw(2, metrics=False))
        run()
        h.sync()
        h.set_wait_limit(0.0)
        with pytest.raises(hot.HotError, match="HOT_ETIMEOUT"):
            for _ in range(50):
                run()
                h.sync()
        h.set_wait_limit(2.0)
        h.set_phase(w.phi0)
        h.set_weights(np.ones(w.M))
        run()
        h.sync()
