"""Tensor mode with a wait limit of zero: the CTAs give up at their first wait that is not over at once,
let what they have in flight finish, and the next synchronising call reports HOT_ETIMEOUT; with a
limit again, the context computes what a new one does, bit for bit."""
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
        with pytest.raises(hot.HotError, match="HOT_ETIMEOUT"):
            h.sync()
        h.set_wait_limit(2.0)
        h.set_phase(w.phi0)
        h.set_weights(np.ones(M))
        h.gsw(3)
        assert all(np.array_equal(a, b) for a, b in zip((h.phase("f32"), *h.fields()), ref))
