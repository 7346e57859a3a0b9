"""GPU: the register-tiled kernels (csrc/tile_kernels.cuh) where their tiles and trap splits have
edges -- one pixel to a few strips of 64 columns, odd and even row counts around a tile's 16 rows,
trap counts around a pair, a team of warps and a reduction group -- in the step, the field of given
phases, the superposition and the adjoint, against the FP64 oracle.

Tolerances as in test_gpu_parity and test_gpu_autograd (|V_m| 1e-4 relative; single-step phases
|S_j| |dphi_j| <= tol sum |c_m|; adjoint tol sum |G_m| / N): every product and sum of the kernels is
FP32 on table entries correct to 2^-24, so tol = 2e-6 holds in all three modes."""
import numpy as np
import pytest

import oracle
from paper_0907_4027_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

REL_V = 1e-4
TOL_S = 2e-6


@pytest.fixture(scope="module")
def hot():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0907_4027_gb300 import _build
    _build.build()
    from paper_0907_4027_gb300 import hot as h
    return h


def rel_err(a, b):
    return np.max(np.abs(np.abs(a) - np.abs(b)) / np.maximum(np.abs(b), 1e-300))


@pytest.mark.parametrize("precision", ["accurate", "fast", "separable"])
@pytest.mark.parametrize("W,H,M", [
    (1, 2, 1), (63, 17, 2), (64, 16, 3), (65, 15, 8), (128, 1, 15), (129, 33, 16), (2, 300, 17),
    (700, 31, 127), (64, 512, 129),   # the unit-phasor state ends at 128 traps
    (1500, 700, 9),                   # teams of 2 and 4 warps, several tiles per team
    (1100, 1000, 20),
])
def test_tiles_match_oracle(hot, W, H, M, precision):
    import torch
    w = wl.random_case(W, H, M, seed=5 * W + 3 * H + M, precision=precision)
    rng = np.random.default_rng(W + H + M)
    coef = rng.normal(size=M) + 1j * rng.normal(size=M)
    phi = rng.uniform(-np.pi, np.pi, w.N).astype(np.float32)
    with hot.Hologram.from_workload(w) as h:
        h.gsw(0)
        V0, _ = h.fields()
        h.gsw(1)
        V1, w1 = h.fields()
        phi1 = h.phase("f32")
        phi_d = torch.tensor(phi, device="cuda")
        V = torch.empty(2 * M, dtype=torch.float32, device="cuda")
        hot.hot_field(h.ctx, phi_d, V)
        grad = torch.empty_like(phi_d)
        G = torch.tensor(np.stack([coef.real, coef.imag], 1).astype(np.float32), device="cuda").reshape(-1)
        hot.hot_field_adjoint(h.ctx, phi_d, G, grad)
        v = V.cpu().numpy().astype(np.float64)
        g = grad.cpu().numpy().astype(np.float64)
        h.superposition(coef)
        sr = h.phase("f32").astype(np.float64)
    assert rel_err(V0, oracle.forward(w.geom, w.xyz, w.phi0)) < REL_V
    r1 = oracle.gsw(w.geom, w.xyz, 1, w.phi0)
    assert rel_err(V1, r1["V"]) < REL_V
    np.testing.assert_allclose(w1, r1["w"], rtol=REL_V)
    # the back-projection from the GPU's own fields (the rounding of a weak |V_m| is not its error)
    for got, c in ((phi1.astype(np.float64), oracle.update_weights(V0, np.ones(M))[1]), (sr, coef)):
        ophi, S = oracle.backproject(w.geom, w.xyz, c, want_S=True)
        d = np.abs(np.angle(np.exp(1j * (got - ophi))))
        assert not (np.abs(S) * d > TOL_S * np.sum(np.abs(c))).any()
    assert rel_err(v[0::2] + 1j * v[1::2], oracle.forward(w.geom, w.xyz, phi.astype(np.float64))) < REL_V
    og = oracle.adjoint(w.geom, w.xyz, phi.astype(np.float64), coef)
    assert np.max(np.abs(g - og)) <= TOL_S * np.sum(np.abs(coef)) / w.N


@pytest.mark.parametrize("precision", ["accurate", "separable"])
def test_tiles_resume_and_persistent_bits(hot, precision):
    """More than 128 traps in teams of 2 warps: resumed calls and the persistent form give the bits
    of one call, as do launches one by one."""
    w = wl.random_case(1300, 900, 130, seed=3, precision=precision)
    out = []
    for mode in ("one", "split", "persistent", "nographs"):
        with hot.Hologram.from_workload(w) as h:
            if mode == "persistent":
                h.use_persistent(True)
            if mode == "nographs":
                h.use_graphs(False)
            if mode == "split":
                h.gsw(1)
                eu = h.gsw(2)
            else:
                eu = h.gsw(3)
            out.append((h.phase("f32"), *h.fields(), eu))
    for p, V, wt, eu in out[1:]:
        assert np.array_equal(out[0][0], p) and np.array_equal(out[0][1], V) and np.array_equal(out[0][2], wt)
        assert eu == out[0][3]
