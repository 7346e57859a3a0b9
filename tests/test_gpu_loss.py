"""hot_intensity_loss over its trap counts: one warp, partly filled warps, several warps, several traps per
thread, with the accumulators in one copy (tensor mode) and in eight (up to 512 traps).  The loss is
formed in 64 bits from the call's own fields, so it has to equal theirs to FP32 rounding; the gradient is
an FP32 sum over the traps, at most M/8 + 8 terms in a row, of products good to some 32 units."""
import numpy as np
import pytest

import oracle
from paper_0907_4027_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0907_4027_gb300 import _build
    _build.build()
    from paper_0907_4027_gb300 import autograd as ag
    from paper_0907_4027_gb300 import hot
    return torch, hot, ag


@pytest.mark.parametrize("precision", ["accurate", "tensor"])
@pytest.mark.parametrize("M", [1, 31, 33, 256, 1024, 1025, 4096])
def test_loss_and_gradient(env, M, precision):
    torch, hot, ag = env
    beta = 10.0
    w = wl.random_case(66, 47, M, seed=M, precision=precision)
    phi0 = w.phi0.astype(np.float32)
    phi = torch.tensor(phi0, device="cuda", requires_grad=True)
    with hot.Hologram.from_workload(w, torch.cuda.current_stream().cuda_stream) as h:
        for _ in range(2):  # the second call starts from cleared accumulators
            phi.grad = None
            loss = ag.intensity_loss(h, phi, beta)
            loss.backward()
        V, _ = h.fields()
        e, u = h.metrics()
    I = np.abs(V) ** 2
    np.testing.assert_allclose(loss.item(), -np.log(I).sum() + beta * I.var(), rtol=2e-7, atol=1e-9)
    np.testing.assert_allclose([e, u], [I.sum(), 1 - (I.max() - I.min()) / (I.max() + I.min())], rtol=1e-6, atol=1e-7)
    G = 2.0 * (-1.0 / I + beta * 2.0 / M * (I - I.mean())) * V
    ref = oracle.adjoint(w.geom, w.xyz, phi0, G)
    bound = (M / 8 + 40) * 2.0 ** -24 * np.abs(G).sum() / w.N
    assert np.max(np.abs(phi.grad.cpu().numpy().reshape(-1) - np.asarray(ref).reshape(-1))) <= bound
