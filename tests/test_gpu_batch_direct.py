"""Batches of the accurate and fast modes evaluate each pair directly, as the direct step kernels
(hot_set_once 0) do: where both cut a hologram into the same sub-tiles (no more 32-pixel row segments
than resident blocks: one segment each) phases, fields and weights are the same bits, call after
call, so that a sequence of batch calls, which goes on from its own state, does not depend on which
kernels single holograms run."""
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


@pytest.mark.parametrize("mode", ["accurate", "fast"])
def test_batches_run_the_direct_step(hot, mode):
    sizes = [(33, 20, 3), (64, 64, 130), (100, 37, 13), (96, 100, 400)]  # the last: traps on few pixels
    ws = [wl.random_case(W, H, M, seed=W + M, precision=mode) for W, H, M in sizes]
    calls = (1, 2, 40)
    ref = []
    for w in ws:
        with hot.Hologram.from_workload(w) as h:
            h.set_once(False)
            ref.append([])
            for k in calls:
                h.gsw(k)
                ref[-1].append((h.phase("f32"), *h.fields()))
    holos = [hot.Hologram.from_workload(w) for w in ws]
    try:
        with hot.Batch(holos) as b:
            b.set_tiling(group_pairs=2.0)  # a group per hologram
            assert b.tiling()["groups"] == len(ws)
            for i, k in enumerate(calls):
                b.gsw(k)
                for h, r in zip(holos, ref):
                    assert all(np.array_equal(x, y) for x, y in zip((h.phase("f32"), *h.fields()), r[i])), (h.M, k)
    finally:
        for h in holos:
            h.close()


@pytest.mark.parametrize("mode", ["accurate", "fast"])
def test_a_lone_member_runs_the_direct_step(hot, mode):
    w = wl.random_case(128, 96, 257, seed=3, precision=mode)
    with hot.Hologram.from_workload(w) as h:
        h.set_once(False)
        h.gsw(5)
        ref = (h.phase("f32"), *h.fields())
    with hot.Hologram.from_workload(w) as h, hot.Batch([h]) as b:
        b.gsw(2)
        h.set_traps(w.xyz)  # the same traps: the batch's tables are built anew
        h.set_phase(w.phi0)
        b.gsw(5)
        assert all(np.array_equal(x, y) for x, y in zip((h.phase("f32"), *h.fields()), ref))
