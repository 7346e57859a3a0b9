"""A change of kernels, mode or tiling for which the device has no memory: the call returns HOT_ENOMEM at
whichever of its allocations is refused (by the library's test seam, on the host), and the context
goes on as it was, bit for bit."""
import ctypes

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


@pytest.fixture
def refuse(hot):
    seam = ctypes.CDLL(hot._LIB_PATH).hot_test_refuse_alloc
    yield seam
    seam(0)


def result(h, w):
    h.set_phase(w.phi0)
    h.set_weights(np.ones(w.M))
    h.gsw(2)
    return (h.phase("f32"), *h.fields())


def same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


CHANGES = {
    "direct": ("fast", lambda h: h.set_once(False)),
    "tile": ("accurate", lambda h: h.set_once(True)),
    "tensor": ("fast", lambda h: h.set_precision("tensor")),
    "separable": ("direct", lambda h: h.set_precision("separable")),
    "leave separable": ("separable off", lambda h: h.set_precision("accurate")),
    "tiling": ("direct", lambda h: h.set_tiling(5, 2, 32)),
    "merge": ("fast", lambda h: h.set_block_merge(4)),
}


@pytest.mark.parametrize("change", CHANGES)
def test_a_refused_change_leaves_the_context_as_it_was(hot, refuse, change):
    start, call = CHANGES[change]
    w = wl.random_case(200, 150, 60, seed=9, precision="separable" if start == "separable off" else "fast")
    with hot.Hologram.from_workload(w) as h:
        if start == "accurate":
            h.set_precision("accurate")
        if start in ("accurate", "direct", "separable off"):
            h.set_once(False)
        ref, tiling = result(h, w), h.tiling()
        nth = 0
        while True:
            nth += 1
            refuse(nth)
            try:
                call(h)
            except hot.HotError as e:
                assert e.status == hot.HOT_ENOMEM and nth < 20
                assert h.tiling() == tiling and same(result(h, w), ref)
            else:
                break
        refuse(0)
        assert nth > 1
        got = result(h, w)
    np.testing.assert_allclose(np.abs(got[1]), np.abs(ref[1]), rtol=1e-4)


def test_a_refused_autotune_leaves_working_kernels(hot, refuse):
    w = wl.random_case(96, 64, 40, seed=3, precision="fast")
    with hot.Hologram.from_workload(w) as h:
        tile = result(h, w)
        for nth in range(1, 28, 3):
            refuse(nth)
            with pytest.raises(hot.HotError, match="HOT_ENOMEM"):
                h.autotune(1)
            assert hot.hot_get_once(h.ctx)["requested"] and same(result(h, w), tile), nth
