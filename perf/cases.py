"""Performance cases of the GSW hologram engine: the calls a user's program makes, over the sizes
this repository's workloads, tests and benchmark use.

Kinds of case (every one through `paper_0907_4027_gb300.hot` / `autograd`):
  gsw    a frame: new trap positions, starting phases, K iterations, phases to a device buffer,
         the traps' fields and weights (`Hologram.set_traps / set_phase / gsw / phase / fields`)
  batch  K more iterations on holograms of uneven size and trap count (`Batch.gsw`)
  sr     a random superposition hologram (`Hologram.superposition`)
  field  the traps' fields of given phases (`hot_field`)
  loss   the differentiable form's loss and gradient (`autograd.intensity_loss`)
  grad   trap fields differentiated through a loss written in PyTorch (`autograd.trap_fields`)

Modes: the accurate mode is a context's default, the fast mode the benchmark's, the separable and
tensor modes are chosen by callers who want their speed.

Starting phases are those of a random superposition hologram, the method's own start (Sec. 5).

Phases are returned as the pixels' complex transmission e^{i phi} in float16: a phase near +-pi may
come out on either side, a pixel where the superposition nearly cancels has no definite phase, and
the modulator resolves 256 levels.  The fields V_m (a sum over every pixel, for each trap) and the
weights are returned in float32, the precision they are computed in.
"""
import math

import numpy as np
import torch

from paper_0907_4027_gb300 import autograd, hot, workloads

BETA = 10.0  # weight of the intensity variance in the differentiable form's loss


def listed():
    return [
        # the smallest call: 16 traps' fields of given phases, as a monitor of a running hologram asks
        {"name": "field16_256", "kind": "field", "W": 256, "H": 256, "M": 16, "traps": "grid", "mode": "accurate"},
        # the paper's SR hologram (Sec. 4, 5): 768^2, a 9 x 9 grid
        {"name": "sr81_768", "kind": "sr", "W": 768, "H": 768, "M": 81, "traps": "grid", "mode": "fast"},
        # the paper's real-time frame: 8 traps on a cube, 5 iterations
        {"name": "cube8_768", "kind": "gsw", "W": 768, "H": 768, "M": 8, "traps": "cube", "mode": "fast", "K": 5},
        # the smallest named workload: 256^2, a 4 x 4 grid, 10 iterations, the default mode
        {"name": "grid16_256", "kind": "gsw", "W": 256, "H": 256, "M": 16, "traps": "grid", "mode": "accurate",
         "K": 10},
        # the benchmark's workload: 512^2, 100 random traps, 30 iterations
        {"name": "rand100_512", "kind": "gsw", "W": 512, "H": 512, "M": 100, "traps": "rand", "mode": "fast",
         "K": 30},
        # an odd-sized modulator region, ragged in both directions
        {"name": "rand37_801x603", "kind": "gsw", "W": 801, "H": 603, "M": 37, "traps": "rand", "mode": "separable",
         "K": 20},
        # more traps than the one-exponential step holds
        {"name": "rand256_1024", "kind": "gsw", "W": 1024, "H": 1024, "M": 256, "traps": "rand", "mode": "fast",
         "K": 30},
        # the largest named workload: a full-HD modulator, 1000 traps, 50 iterations, the default mode
        {"name": "rand1000_1920", "kind": "gsw", "W": 1920, "H": 1152, "M": 1000, "traps": "rand", "mode": "accurate",
         "K": 50},
        # the same on the tensor cores
        {"name": "rand1000_1920_tensor", "kind": "gsw", "W": 1920, "H": 1152, "M": 1000, "traps": "rand",
         "mode": "tensor", "K": 50},
        # one optimiser step's loss and gradient in the differentiable configuration
        {"name": "loss256_1024", "kind": "loss", "W": 1024, "H": 1024, "M": 256, "traps": "rand", "mode": "fast"},
        # the same through torch.autograd with the loss in PyTorch
        {"name": "grad100_512", "kind": "grad", "W": 512, "H": 512, "M": 100, "traps": "rand", "mode": "accurate"},
        # 8 holograms of the batched configuration's sizes and trap counts, 5 iterations
        {"name": "batch8", "kind": "batch", "count": 8, "wmax": 1920, "M": 2000, "mode": "fast", "K": 5},
    ]


def _spread(rng, lo, hi):
    """An integer of [lo, hi], uniform over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["gsw", "gsw", "gsw", "gsw", "batch", "sr", "field", "loss", "grad"])
    mode = rng.choice(["accurate", "fast", "separable"])
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(2, 16), "wmax": _spread(rng, 128, 1024), "M": _spread(rng, 16, 1000),
                "mode": mode, "K": rng.randint(1, 20)}
    W, H = _spread(rng, 128, 1920), _spread(rng, 128, 1152)
    traps = rng.choice(["grid", "rand", "rand", "rand"])
    M = rng.randint(2, 9) ** 2 if traps == "grid" else _spread(rng, 4, 1500)
    c = {"kind": kind, "W": W, "H": H, "M": M, "traps": traps, "mode": mode}
    if kind == "gsw":
        c["mode"] = rng.choice([mode, mode, mode, "tensor"])
        c["K"] = max(1, min(_spread(rng, 1, 50), int(5e10 / (W * H * M))))
    return c


# ---- inputs ------------------------------------------------------------------------------------

def _traps(case, rng):
    """(M, 3) trap positions in metres, moved a little from frame to frame."""
    M = case["M"]
    if case["traps"] == "grid":
        xyz = workloads.square_grid(int(round(math.sqrt(M))), 4.0)
    elif case["traps"] == "cube":
        xyz = workloads.cube(5.0)
    else:
        xy, z = (60.0, 15.0) if M > 128 else (40.0, 10.0)
        return workloads.random_traps(M, xy, z, int(rng.integers(1 << 30)))
    return xyz + rng.uniform(-0.2e-6, 0.2e-6, (1, 3))


def _members(case, rng):
    """Members of a batch: sizes in the ratios of 512^2 : 1024^2 : 1920 x 1152, M ~ U{8..M}."""
    wmax = case["wmax"]
    sizes = [(wmax * 512 // 1920, wmax * 512 // 1920), (wmax * 1024 // 1920, wmax * 1024 // 1920),
             (wmax, wmax * 1152 // 1920)]
    shape = np.random.default_rng(case["count"])  # the sizes belong to the case, the positions to the seed
    out = []
    for i in range(case["count"]):
        W, H = sizes[i % 3]
        M = int(shape.integers(8, case["M"] + 1))
        out.append((W, H, workloads.random_traps(M, 60.0, 15.0, int(rng.integers(1 << 30)))))
    return out


def _parts(W, H, xyz):
    """Eq. 2 in 64 bits: unit phasors of the column parts (M, W) and of the row parts (M, H)."""
    lin = workloads.PITCH / (workloads.WAVELENGTH * workloads.FOCAL)
    quad = workloads.PITCH ** 2 / (2.0 * workloads.WAVELENGTH * workloads.FOCAL ** 2)
    t = torch.as_tensor(xyz, dtype=torch.float64, device="cuda")
    x = torch.arange(W, dtype=torch.float64, device="cuda") - W // 2
    y = torch.arange(H, dtype=torch.float64, device="cuda") - H // 2
    a, b, c = t[:, 0:1] * lin, t[:, 1:2] * lin, t[:, 2:3] * quad
    out = []
    for turns in (a * x + c * x * x, b * y + c * y * y):
        turns = turns - torch.round(turns)
        out.append(torch.polar(torch.ones_like(turns), 2.0 * math.pi * turns))
    return out


def _superpose(X, Y, coef):
    """sum_m c_m e^{i Delta_j^m} as an (H, W) array."""
    return (coef[:, None] * Y).T @ X


def _unit_coefficients(M, rng):
    return np.exp(1j * rng.uniform(-np.pi, np.pi, M))


def _start_phases(W, H, xyz, rng):
    """float32 device phases of the random superposition hologram a run starts from."""
    X, Y = _parts(W, H, xyz)
    coef = torch.as_tensor(_unit_coefficients(len(xyz), rng), device="cuda")
    return _superpose(X, Y, coef).angle().to(torch.float32).reshape(-1).contiguous()


def _inputs(case, seed):
    """Everything that depends on the seed."""
    rng = np.random.default_rng([int(seed), 17])
    if case["kind"] == "batch":
        members = _members(case, rng)
        return {"members": members, "phi": [_start_phases(W, H, xyz, rng) for W, H, xyz in members]}
    xyz = _traps(case, rng)
    W, H = case["W"], case["H"]
    if case["kind"] == "sr":
        return {"xyz": xyz, "coef": _unit_coefficients(len(xyz), rng)}
    phi = _start_phases(W, H, xyz, rng)
    if case["kind"] in ("loss", "grad"):  # in the course of an optimisation: away from the start
        phi = phi + torch.as_tensor(rng.normal(0.0, 0.3, W * H).astype(np.float32), device="cuda")
    return {"xyz": xyz, "phi": phi}


def _hologram(W, H, mode):
    return hot.Hologram(W, H, workloads.PITCH, workloads.WAVELENGTH, workloads.FOCAL, precision=mode)


def prepare(case, seed):
    s = {"case": case, **_inputs(case, seed)}
    if case["kind"] == "batch":
        s["holo"] = [_hologram(W, H, case["mode"]) for W, H, _ in s["members"]]
        for h, (_, _, xyz), phi in zip(s["holo"], s["members"], s["phi"]):
            h.set_traps(xyz)
            h.set_phase(phi)
        s["batch"] = hot.Batch(s["holo"])
        s["out"] = torch.empty(sum(h.N for h in s["holo"]), dtype=torch.float32, device="cuda")
        return s
    h = s["holo"] = _hologram(case["W"], case["H"], case["mode"])
    h.set_traps(s["xyz"])
    s["out"] = torch.empty(h.N, dtype=torch.float32, device="cuda")
    s["V"] = torch.empty(2 * h.M, dtype=torch.float32, device="cuda")
    if case["kind"] in ("loss", "grad"):
        s["phi"] = s["phi"].requires_grad_(True)
    return s


def _transmission(phi):
    """e^{i phi} of device phases, (N, 2) float16."""
    return torch.view_as_real(torch.polar(torch.ones_like(phi), phi)).half()


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "gsw":
        h = s["holo"]
        h.set_traps(s["xyz"])
        h.set_phase(s["phi"])
        e, u = h.gsw(case["K"])
        h.phase("f32", out=s["out"])
        V, w = h.fields()
        return {"field": _transmission(s["out"]), "V": V.astype(np.complex64), "w": w.astype(np.float32), "e": e, "u": u}
    if kind == "batch":
        s["batch"].gsw(case["K"])
        at, V, w = 0, [], []
        for h in s["holo"]:
            h.phase("f32", out=s["out"][at:at + h.N])
            at += h.N
            Vh, wh = h.fields()
            V.append(Vh.astype(np.complex64))
            w.append(wh.astype(np.float32))
        return {"field": _transmission(s["out"]), "V": V, "w": w}
    if kind == "sr":
        s["holo"].superposition(s["coef"])
        s["holo"].phase("f32", out=s["out"])
        return _transmission(s["out"])
    if kind == "field":
        hot.hot_field(s["holo"].ctx, s["phi"], s["V"])
        return s["V"]
    s["phi"].grad = None
    if kind == "loss":
        loss = autograd.intensity_loss(s["holo"], s["phi"], BETA)
        loss.backward()
        return {"loss": loss.detach(), "grad": s["phi"].grad}
    V = autograd.trap_fields(s["holo"], s["phi"])
    loss = autograd.trap_intensity_loss(V, BETA)
    loss.backward()
    return {"V": V.detach(), "loss": loss.detach(), "grad": s["phi"].grad}


# ---- what a pass cannot do without -----------------------------------------------------------

def work(case):
    """Per pixel-trap pair one complex multiply-add (8 flops) forward and one back; the phases and
    the traps' values read once and written once."""
    if case["kind"] == "batch":
        parts = [(W * H, len(xyz)) for W, H, xyz in _members(case, np.random.default_rng(0))]
        return {"flops": sum(8.0 * N * M * (2 * case["K"] + 1) for N, M in parts),
                "bytes": sum(8.0 * N + 12.0 * N + 48.0 * M for N, M in parts)}
    N, M = case["W"] * case["H"], case["M"]
    steps = {"gsw": 2 * case.get("K", 0) + 1, "sr": 1, "field": 1, "loss": 2, "grad": 2}[case["kind"]]
    per_pixel = {"gsw": 4 + 4 + 4, "sr": 4 + 4, "field": 4, "loss": 4 + 4, "grad": 4 + 4}[case["kind"]]
    return {"flops": 8.0 * N * M * steps, "bytes": float(per_pixel * N + 48 * M)}


# ---- the same in 64 bits ------------------------------------------------------------------------

def _fields(X, Y, u):
    """V_m = (1/N) sum_j u_j e^{-i Delta_j^m} (Eq. 1)."""
    return ((u @ X.conj().T) * Y.conj().T).sum(0) / u.numel()


def _gsw(W, H, xyz, phi, K, w=None):
    X, Y = _parts(W, H, xyz)
    phi = phi.to(torch.float64).reshape(H, W)
    u = torch.polar(torch.ones_like(phi), phi)
    w = torch.ones(len(xyz), dtype=torch.float64, device="cuda") if w is None else w
    V = _fields(X, Y, u)
    for _ in range(K):
        w = w * V.abs().mean() / V.abs()
        S = _superpose(X, Y, w * V / V.abs())
        u = S / S.abs()
        V = _fields(X, Y, u)
    return torch.view_as_real(u.reshape(-1)), V, w


def exact(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "gsw":
        u, V, w = _gsw(case["W"], case["H"], s["xyz"], s["phi"], case["K"])
        I = V.abs() ** 2
        return {"field": u, "V": V, "w": w, "e": I.sum(),
                "u": 1.0 - (I.max() - I.min()) / (I.max() + I.min())}
    if kind == "batch":
        got = [_gsw(W, H, xyz, phi, case["K"]) for (W, H, xyz), phi in zip(s["members"], s["phi"])]
        return {"field": torch.cat([g[0] for g in got]), "V": [g[1] for g in got], "w": [g[2] for g in got]}
    X, Y = _parts(case["W"], case["H"], s["xyz"])
    if kind == "sr":
        S = _superpose(X, Y, torch.as_tensor(s["coef"], device="cuda")).reshape(-1)
        return torch.view_as_real(S / S.abs())
    phi = s["phi"].to(torch.float64).reshape(case["H"], case["W"])
    u = torch.polar(torch.ones_like(phi), phi)
    V = _fields(X, Y, u)
    if kind == "field":
        return torch.view_as_real(V).reshape(-1)
    I = V.abs() ** 2
    loss = -torch.log(I).sum() + BETA * I.var(correction=0)
    G = 2.0 * (-1.0 / I + BETA * (2.0 / len(I)) * (I - I.mean())) * V
    grad = (u.conj() * _superpose(X, Y, G)).imag.reshape(-1) / phi.numel()
    if kind == "loss":
        return {"loss": loss, "grad": grad}
    return {"V": V, "loss": loss, "grad": grad}
