"""A batch on a stream of its own starts after what its members queued on theirs: weights, traps,
phases and superpositions that the GPU has not reached yet when hot_batch_gsw is called (and when
its autotuner saves the state)."""
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


def change(h, what, rng):
    if what == "superposition":
        h.superposition(np.exp(1j * rng.uniform(-3, 3, h.M)))
    elif what == "weights":
        h.set_weights(rng.uniform(0.5, 2.0, h.M))
    else:
        h.set_traps(rng.uniform(-4e-5, 4e-5, (h.M, 3)))


@pytest.mark.parametrize("precision", ["accurate", "separable", "tensor"])
@pytest.mark.parametrize("what", ["superposition", "weights", "traps"])
def test_batch_waits_for_its_members(hot, what, precision):
    import torch
    ws = [wl.random_case(W, H, M, seed=M, precision=precision) for W, H, M in ((100, 37, 13), (256, 128, 40))]
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    busy = hot.Hologram.from_workload(wl.random_case(1024, 1024, 200, seed=1, precision="fast"), mine.cuda_stream)

    def run(behind):
        holos = [hot.Hologram.from_workload(w, mine.cuda_stream) for w in ws]
        out = []
        with hot.Batch(holos, other.cuda_stream) as b:
            for turn in range(2):  # the second run replays the first one's graph
                rng = np.random.default_rng(5 + turn)
                torch.cuda.synchronize()
                if behind:
                    busy.gsw(100, metrics=False)  # some 10 ms
                for h in holos:
                    change(h, what, rng)
                if not behind:
                    torch.cuda.synchronize()
                b.gsw(2)
                other.synchronize()
                out += [(h.phase("f32"), *h.fields()) for h in holos]
        for h in holos:
            h.close()
        return out

    busy.gsw(100)
    ref, got = run(False), run(True)
    busy.close()
    for r, g in zip(ref, got):
        assert all(np.array_equal(x, y) for x, y in zip(r, g))


def test_autotuner_saves_what_its_members_queued(hot):
    import torch
    w = wl.random_case(100, 37, 13, seed=1, precision="separable")
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    busy = hot.Hologram.from_workload(wl.random_case(1024, 1024, 200, seed=1, precision="fast"), mine.cuda_stream)
    busy.gsw(100)
    coef = np.exp(1j * np.arange(13.0))
    with busy, hot.Hologram.from_workload(w, mine.cuda_stream) as h, hot.Batch([h], other.cuda_stream) as b:
        h.superposition(coef)
        ref = h.phase("f32")
        h.set_phase(w.phi0)
        torch.cuda.synchronize()
        busy.gsw(100, metrics=False)
        h.superposition(coef)
        b.autotune(1)
        assert np.array_equal(h.phase("f32"), ref)
