"""Groups of one hologram in a batch: they run hot_gsw's own tiles and teams, so above 128 traps (where
a call's state is the phases) their results are the bits of hot_gsw, beside groups of several holograms,
after a resumed call and after the member's own tiles were rebuilt; a tiling that is asked for is
kept to."""
import numpy as np
import pytest

import oracle
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


@pytest.mark.parametrize("mode", ["accurate", "separable"])
def test_lone_groups_equal_single_runs(hot, mode):
    sizes = [(65, 33, 129), (801, 660, 131), (640, 301, 400)]  # group_pairs below: three groups
    ws = [wl.random_case(W, H, M, seed=W + M, precision=mode) for W, H, M in sizes]
    ref = []
    for w in ws:
        with hot.Hologram.from_workload(w) as h:
            h.gsw(3)
            ref.append((h.phase("f32"), *h.fields()))
    holos = [hot.Hologram.from_workload(w) for w in ws]
    try:
        with hot.Batch(holos) as b:
            b.set_tiling(group_pairs=1.0)
            b.gsw(2)
            holos[1].set_once(False)  # drops the context's own tiles: the batch has its own
            holos[1].set_once(True)
            b.gsw(1)
            got = [(h.phase("f32"), *h.fields()) for h in holos]
            tiled = []
            b.set_tiling(rows=5, group_pairs=1.0)
            for h, w in zip(holos, ws):
                h.set_phase(w.phi0)
                h.set_weights(np.ones(w.M))
            b.gsw(1)
            tiled = [h.fields()[0] for h in holos]
    finally:
        for h in holos:
            h.close()
    for (p0, V0, w0), (p1, V1, w1) in zip(ref, got):
        assert np.array_equal(p0, p1) and np.array_equal(V0, V1) and np.array_equal(w0, w1)
    for V, w in zip(tiled, ws):
        oV = oracle.gsw(w.geom, w.xyz, 1, w.phi0)["V"]
        assert np.max(np.abs(np.abs(V) - np.abs(oV)) / np.abs(oV)) < 1e-4
