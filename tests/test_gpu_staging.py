"""GPU: the pinned staging of a context's small transfers (traps, weights, coefficients, fields,
metrics): calls queued one after the other without a synchronisation each use their own values, the
timeout of a bounded wait is still reported by every call that reads back, and a captured stream is
refused."""
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


@pytest.mark.parametrize("M", [1, 33, 700])
def test_queued_calls_keep_their_values(hot, M):
    """20 frames queued back to back (new traps, weights and coefficients each) on a busy stream equal
    the same frames run alone, bit for bit."""
    import torch
    W, H, n = 300, 200, 20
    rng = np.random.default_rng(M)
    xyz = [wl.random_traps(M, 40.0, 10.0, seed=i) for i in range(n)]
    w = rng.uniform(0.5, 2.0, (n, M))
    coef = np.exp(1j * rng.uniform(-np.pi, np.pi, (n, M)))
    stream = torch.cuda.Stream()

    def frame(h, i, out):
        h.set_traps(xyz[i])
        h.set_weights(w[i])
        h.superposition(coef[i])
        h.gsw(1, metrics=False)
        h.phase("f32", out=out)

    with hot.Hologram(W, H, wl.PITCH, wl.WAVELENGTH, wl.FOCAL, stream.cuda_stream, "fast") as h:
        got = [torch.empty(W * H, device="cuda") for _ in range(n)]
        h.set_traps(xyz[0])
        h.gsw(200, metrics=False)  # the stream is behind the host
        for i in range(n):
            frame(h, i, got[i])
        V, wt = h.fields()
        eu = h.metrics()
        ref = torch.empty(W * H, device="cuda")
        for i in range(n):
            frame(h, i, ref)
            h.sync()
            assert torch.equal(ref, got[i]), i
        Vr, wr = h.fields()
        assert np.array_equal(V, Vr) and np.array_equal(wt, wr) and eu == h.metrics()
        np.testing.assert_allclose(eu[0], np.sum(np.abs(V) ** 2), rtol=1e-5)


@pytest.mark.parametrize("read", ["fields", "metrics", "sync"])
def test_wait_timeout_reaches_the_reading_call(hot, read):
    w = wl.random_case(128, 64, 9, seed=6, precision="fast")
    with hot.Hologram.from_workload(w) as h:
        h.use_persistent(True)
        h.set_wait_limit(0.0)
        h.gsw(5, metrics=False)
        with pytest.raises(hot.HotError, match="HOT_ETIMEOUT"):
            getattr(h, read)()
        h.set_wait_limit(2.0)
        h.set_phase(w.phi0)
        h.set_weights(np.ones(w.M))
        h.gsw(1)
        h.fields()


def test_captured_stream_is_refused(hot):
    import torch
    w = wl.random_case(64, 32, 5, seed=1, precision="fast")
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        with hot.Hologram.from_workload(w, stream.cuda_stream) as h:
            h.superposition(np.ones(5))
            h.sync()
            g = torch.cuda.CUDAGraph()
            x = torch.zeros(4, device="cuda")
            with torch.cuda.graph(g, stream=stream):
                for call in (lambda: h.set_traps(w.xyz), lambda: h.set_weights(np.ones(5)),
                             lambda: h.superposition(np.ones(5))):
                    with pytest.raises(hot.HotError, match="HOT_ECUDA"):
                        call()
                x += 1
            h.gsw(1)
