"""Performance cases of the solver: the work its users have it do, through the
public entry points, with the same results in 64 bits beside them.

A case is a dict of plain values; `kind` names the call sequence:

  step         Solver.step(steps), then Solver.populations() into pinned FP32 memory
               (a run between two checkpoints); FP32, FP16 or BF16 storage
  diagnostics  Solver.diagnostics() and Solver.profile() of a state (the energy-budget
               evaluation that a run makes every 100 steps)
  ensemble     Ensemble.step(steps) of realisations of two grid sizes, mixed couplings
               and storage types, then every member's populations
  noalloc      one lbm_step_noalloc on device arrays (the embedding interface)
  infer        Cnn.infer: the closure network on the tensor cores
  train        lbm_cnn_loss_grad: forward and backward of one training sample
  closure      Closure.advance: corrected intervals of the 2x-coarsened run, then the
               coarse run's populations

Every state starts from a seeded Rayleigh-Taylor flow: a perturbed tanh interface
(the workloads' masses 1.0 / 0.9 and 8 % minority) with a seeded velocity field.
"""
from __future__ import annotations

import ctypes as C
import math

import numpy as np
import torch

from paper_2101_04847_gb300 import lbm

CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
MASS_A, MASS_B, CROP = 1.0, 0.9, 10
CNN_SHAPES = ((32, 4, 3, 3), (32,), (32, 32, 3, 3), (32,), (4, 32, 3, 3), (4,))
CLOSURE_INTERVAL, CLOSURE_MODE = 10, 4
# normalisation of a trained closure at these workloads: means and scales of
# (rho_A, rho_B, u_x, u_y), and the size of its corrections
IN_MEAN, IN_SCALE, OUT_SCALE = (0.54, 0.49, 0.0, 0.0), (0.46, 0.41, 0.01, 0.01), (1e-3, 1e-3, 1e-4, 1e-4)


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _flow(**kw) -> dict:
    return dict(dict(G=1.4, g=1e-5, minority=0.08, gravity_mode=0, wall_mode=0), **kw)


def listed() -> list[dict]:
    return [
        # the small validation grid: a launch has a few thousand sites per SM at most,
        # so what a step costs is its latency
        _flow(name="step_128x256_f32", kind="step", nx=128, ny=256, steps=100, storage="f32"),
        # the measured workload, in each storage precision
        _flow(name="step_1024x2048_f32", kind="step", nx=1024, ny=2048, steps=200, storage="f32"),
        _flow(name="step_1024x2048_f16", kind="step", nx=1024, ny=2048, steps=200, storage="f16"),
        # the full-size production grid, FP32 and 16-bit storage: more steps to a
        # checkpoint, whose 3.6 GB cross the host link
        _flow(name="step_10000x5000_f32", kind="step", nx=10000, ny=5000, steps=500, storage="f32"),
        _flow(name="step_10000x5000_f16", kind="step", nx=10000, ny=5000, steps=500, storage="f16"),
        # an odd, ragged grid: the miscible variant in BF16 with mirror walls
        _flow(name="step_1501x999_bf16", kind="step", nx=1501, ny=999, steps=200, storage="bf16", G=0.0, minority=0.0,
              wall_mode=1),
        # the evaluation made every 100 steps of the measured workload
        _flow(name="diagnostics_1024x2048", kind="diagnostics", nx=1024, ny=2048, storage="f32"),
        # ten realisations per experiment, uneven grids, couplings and storage types
        dict(name="ensemble_10", kind="ensemble", members=10, nx=512, ny=1024, nx2=1024, ny2=2048, steps=200),
        # a host application's own time loop: one step per call on its arrays
        _flow(name="noalloc_512x1024", kind="noalloc", nx=512, ny=1024),
        # the network on the coarse grid of the full-size run
        dict(name="infer_5000x2500", kind="infer", nx=5000, ny=2500),
        # one training sample of the 1024x2048 fine runs
        dict(name="train_512x1024", kind="train", nx=512, ny=1024),
        # the learned closure in production: ten corrected intervals of the coarse run
        _flow(name="closure_1024x2048", kind="closure", nx=1024, ny=2048, intervals=10),
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def _grid(rng, lo: int, hi: int, most: int) -> tuple[int, int]:
    while True:
        nx, ny = _log_int(rng, lo, hi), _log_int(rng, lo, hi)
        if nx * ny <= most:
            return nx, ny


def draw(rng) -> dict:
    kind = rng.choice(["step"] * 5 + ["diagnostics"] * 2 + ["noalloc"] * 2 + ["ensemble", "infer", "train", "closure"])
    if kind in ("infer", "train"):
        nx, ny = _grid(rng, 24, 4096 if kind == "infer" else 1024, 8 << 20)
        return dict(kind=kind, nx=nx, ny=ny)
    if kind == "ensemble":
        nx, ny = _grid(rng, 48, 1024, 1 << 19)
        nx2, ny2 = _grid(rng, 48, 2048, 1 << 21)
        return dict(kind=kind, members=rng.randint(2, 12), nx=nx, ny=ny, nx2=nx2, ny2=ny2, steps=rng.randint(20, 120))
    G = rng.choice([0.0, 1.2, 1.4])
    flow = _flow(kind=kind, G=G, minority=0.0 if G == 0.0 else 0.08, gravity_mode=rng.choice([0, 0, 1]),
                 wall_mode=rng.choice([0, 1]))
    if kind == "noalloc":
        nx, ny = _grid(rng, 32, 4096, 1 << 20)
        return dict(flow, nx=nx, ny=ny)
    if kind == "closure":
        nx, ny = _grid(rng, 48, 2048, 1 << 21)
        return dict(flow, nx=nx, ny=ny, intervals=rng.randint(1, 6))
    nx, ny = _grid(rng, 32, 8192, 1 << 24)
    flow = dict(flow, nx=nx, ny=ny, storage=rng.choice(["f32", "f16", "bf16"]))
    return flow if kind == "diagnostics" else dict(flow, steps=rng.randint(20, 200))


def _members(case: dict) -> list[dict]:
    """The realisations of an ensemble case: small and large grids in turn, the three
    couplings, FP32 and FP16 storage."""
    out = []
    for i in range(case["members"]):
        G = (1.4, 1.2, 0.0)[i % 3]
        big = i % 2 == 1
        out.append(_flow(nx=case["nx2"] if big else case["nx"], ny=case["ny2"] if big else case["ny"], G=G,
                         minority=0.0 if G == 0.0 else 0.08, storage="f16" if (i // 2) % 2 else "f32"))
    return out


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _populations(case: dict, seed: int, nx: int, ny: int) -> torch.Tensor:
    """FP32 post-streaming populations [2, 9, ny, nx] on the GPU: the equilibrium of a
    tanh interface at ny / 2, displaced by 8 seeded modes, in a seeded velocity field of
    a few vortices with speeds up to about 0.02."""
    r = np.random.default_rng(seed)
    a, th = r.uniform(size=8), r.uniform(0, 2 * math.pi, size=8)
    xs = np.arange(nx)
    eta = sum(a[m] * np.sin(2 * math.pi * (m + 1) * xs / nx + th[m]) for m in range(8))
    y0 = torch.tensor(ny / 2 + min(8.0, ny / 16) * eta / np.max(np.abs(eta)), device="cuda")
    y = torch.arange(ny, dtype=torch.float64, device="cuda")[:, None]
    x = torch.arange(nx, dtype=torch.float64, device="cuda")[None, :]
    H = 0.5 * (1.0 + torch.tanh((y - y0[None, :]) / 1.5))
    eps = case["minority"]
    rho = (MASS_A * (eps + (1 - eps) * H), MASS_B * (eps + (1 - eps) * (1 - H)))
    ux, uy = torch.zeros_like(H), torch.zeros_like(H)
    for kx, ky, u, p in zip(r.integers(1, 4, 4), r.integers(1, 4, 4), r.uniform(-0.01, 0.01, 4), r.uniform(0, 6.28, 4)):
        px, py = 2 * math.pi * kx * x / nx + p, math.pi * ky * (y + 0.5) / ny
        ux += u * torch.cos(px) * torch.cos(py)
        uy += u * torch.sin(px) * torch.sin(py)
    usq = 1.5 * (ux * ux + uy * uy)
    f = torch.empty((2, 9, ny, nx), dtype=torch.float32, device="cuda")
    for i in range(9):
        cu = CX[i] * ux + CY[i] * uy
        q = W[i] * (1 + 3 * cu + 4.5 * cu * cu - usq)
        for s in range(2):
            f[s, i] = rho[s] * q
    return f


def _pinned(f: torch.Tensor) -> torch.Tensor:
    h = torch.empty(f.shape, dtype=f.dtype, pin_memory=True)
    h.copy_(f)
    return h


def _params(case: dict, nx: int, ny: int, **kw):
    return lbm.default_params(nx=nx, ny=ny, tau_A=1.0, tau_B=1.0, G=case["G"], mass_A=MASS_A, mass_B=MASS_B, g=case["g"],
                              minority=case["minority"], gravity_mode=case["gravity_mode"], wall_mode=case["wall_mode"],
                              crop_rows=min(CROP, ny // 4), **kw)


def _network(seed: int) -> np.ndarray:
    """He-scaled weights and small biases, as a trained network has."""
    r = np.random.default_rng(seed + 7)
    return np.concatenate([r.normal(0.0, math.sqrt(2.0 / (s[1] * 9)) if len(s) == 4 else 0.1, size=s).ravel()
                           for s in CNN_SHAPES]).astype(np.float32)


def _images(case: dict, seed: int) -> tuple[torch.Tensor, torch.Tensor]:
    """Normalised network input and training target [4, ny, nx]: smooth fields of order 1
    (densities saturated in the bulks) with noise on them."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    nx, ny = case["nx"], case["ny"]
    f = _populations(dict(minority=0.08), seed, nx, ny)
    rho = f.sum(1)
    m = [sum(c[i] * f[:, i].sum(0) for i in range(9)) / rho.sum(0) for c in (CX, CY)]
    x = torch.stack([(v - IN_MEAN[k]) / IN_SCALE[k] for k, v in enumerate((rho[0], rho[1], *m))]).float()
    noise = torch.randn((8, ny, nx), generator=g, device="cuda")
    return (x + 0.1 * noise[:4]).contiguous(), noise[4:].contiguous()


def prepare(case: dict, seed: int):
    kind, nx, ny = case["kind"], case["nx"], case["ny"]
    if kind in ("step", "diagnostics"):
        host = _pinned(_populations(case, seed, nx, ny)).numpy()
        solver = lbm.Solver(_params(case, nx, ny, storage=case["storage"]))
        solver.set_populations(host)
        return dict(case=case, solver=solver, host=host)
    if kind == "ensemble":
        members = _members(case)
        ens = lbm.Ensemble([_params(m, m["nx"], m["ny"], storage=m["storage"]) for m in members])
        host = [_pinned(_populations(m, seed * 100 + i, m["nx"], m["ny"])).numpy() for i, m in enumerate(members)]
        for h, s in zip(host, ens.members):
            s.set_populations(h)
        return dict(case=case, ens=ens, host=host)
    if kind == "noalloc":
        f = _populations(case, seed, nx, ny)
        return dict(case=case, params=_params(case, nx, ny), f=f, out=torch.empty_like(f), lib=lbm.load_library())
    if kind == "closure":
        fine = _params(dict(case, g=case["g"] / 8), 2 * nx, 2 * ny)
        closure = lbm.Closure(fine, interval=CLOSURE_INTERVAL, seed=0)
        closure.set_params(_network(seed))
        closure.set_normalisation(IN_MEAN, IN_SCALE, OUT_SCALE)
        _, coarse = closure.solvers()
        host = _pinned(_populations(case, seed, nx, ny)).numpy()
        coarse.set_populations(host)
        return dict(case=case, closure=closure, coarse=coarse, host=host)
    x, t = _images(case, seed)
    cnn = lbm.Cnn(nx, ny)
    p = torch.from_numpy(_network(seed)).cuda()
    state = dict(case=case, cnn=cnn, params=p, x=x, lib=lbm.load_library())
    if kind == "infer":
        return dict(state, y=torch.empty_like(x))
    return dict(state, t=t, grad=torch.empty_like(p))


def _checked(status: int):
    if status != lbm.LBM_OK:
        raise lbm.LbmError(status, "call", lbm.load_library().lbm_last_error().decode())


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "step":
        state["solver"].step(case["steps"])
        return state["solver"].populations(out=state["host"])
    if kind == "diagnostics":
        return dict(terms=state["solver"].diagnostics(), profile=state["solver"].profile())
    if kind == "ensemble":
        state["ens"].step(case["steps"])
        return [m.populations(out=h) for m, h in zip(state["ens"].members, state["host"])]
    if kind == "noalloc":
        stream = torch.cuda.current_stream().cuda_stream
        _checked(state["lib"].lbm_step_noalloc(C.byref(state["params"]), C.c_void_p(state["f"].data_ptr()),
                                               C.c_void_p(state["out"].data_ptr()), C.c_void_p(stream)))
        return state["out"]
    if kind == "closure":
        state["closure"].advance(case["intervals"], CLOSURE_MODE)
        return state["coarse"].populations(out=state["host"])
    if kind == "infer":
        state["cnn"].infer(state["params"], state["x"], state["y"])
        return state["y"]
    cnn, loss = state["cnn"], C.c_double()
    stream = torch.cuda.current_stream().cuda_stream
    _checked(state["lib"].lbm_cnn_loss_grad(
        *(C.c_void_p(state[k].data_ptr()) for k in ("params", "x", "t")), cnn.nx, cnn.ny, C.c_void_p(cnn.ws.data_ptr()),
        cnn.ws.numel(), C.c_void_p(stream), C.byref(loss), C.c_void_p(state["grad"].data_ptr())))
    return dict(loss=loss.value, grad=state["grad"])


def work(case: dict) -> dict:
    """A time step reads and writes 18 stored populations per site; the diagnostics read
    them; the network reads and writes its images (hidden layers stay on chip at best)
    and multiplies 11520 weights per pixel, three times that with the backward passes."""
    kind, n = case["kind"], case["nx"] * case["ny"]
    if kind == "step":
        return dict(bytes=36 * n * (4 if case["storage"] == "f32" else 2) * case["steps"], flops=300 * n * case["steps"])
    if kind == "diagnostics":
        return dict(bytes=18 * n * (4 if case["storage"] == "f32" else 2), flops=500 * n)
    if kind == "ensemble":
        sites = [(m["nx"] * m["ny"], 4 if m["storage"] == "f32" else 2) for m in _members(case)]
        return dict(bytes=case["steps"] * sum(36 * s * b for s, b in sites), flops=300 * case["steps"] * sum(s for s, _ in sites))
    if kind == "noalloc":
        return dict(bytes=144 * n, flops=300 * n)
    if kind == "closure":
        k = case["intervals"]
        return dict(bytes=k * n * 144 * (CLOSURE_INTERVAL + 1), flops=k * n * (300 * CLOSURE_INTERVAL + 23040))
    return dict(bytes=(32 if kind == "infer" else 32 + 16) * n, flops=23040 * n * (1 if kind == "infer" else 3))


# ---------------------------------------------------------------------------
# the same results in 64 bits, plain torch on the GPU
# ---------------------------------------------------------------------------
def _neighbour_sum(r: torch.Tensor, mirror: bool) -> tuple[torch.Tensor, torch.Tensor]:
    """sum_i w_i r(x + c_i) c_i, x periodic, beyond the walls 0 or the wall row's value."""
    lo, hi = (r[:1], r[-1:]) if mirror else (torch.zeros_like(r[:1]),) * 2
    p = torch.cat([lo, r, hi])
    sx, sy = torch.zeros_like(r), torch.zeros_like(r)
    for i in range(1, 9):
        v = torch.roll(p[1 + CY[i]:1 + CY[i] + r.shape[0]], -CX[i], 1) * W[i]
        sx += CX[i] * v
        sy += CY[i] * v
    return sx, sy


def _accelerations(rho: torch.Tensor, case: dict) -> list[tuple[torch.Tensor, torch.Tensor]]:
    sign = (-1.0, 1.0 if case["gravity_mode"] == 0 else -1.0)
    out = []
    for s in range(2):
        sx, sy = _neighbour_sum(rho[1 - s], case["wall_mode"] == 1)
        out.append((-case["G"] * sx, -case["G"] * sy + sign[s] * case["g"]))
    return out


def _momenta(f: torch.Tensor) -> tuple[torch.Tensor, torch.Tensor]:
    """sum_{s,i} f_i^s c_i."""
    return tuple(sum(c[i] * (f[0, i] + f[1, i]) for i in range(1, 9) if c[i]) for c in (CX, CY))


def _equilibrium(i: int, rho, ux, uy):
    cu = CX[i] * ux + CY[i] * uy
    return W[i] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (ux * ux + uy * uy))


def _exact_step(f: torch.Tensor, case: dict) -> torch.Tensor:
    """One forced BGK step at tau = 1 (the collision replaces f by the equilibrium at
    u + a_s), streaming, half-way bounce-back."""
    rho = f.sum(1)
    jx, jy = _momenta(f)
    rt = rho[0] + rho[1]
    jx /= rt
    jy /= rt
    new = torch.empty_like(f)
    for s, (ax, ay) in enumerate(_accelerations(rho, case)):
        vx, vy = jx + ax, jy + ay
        for i in range(9):
            o = _equilibrium(i, rho[s], vx, vy)
            m = torch.roll(o, CX[i], 1) if CX[i] else o
            if CY[i] == 0:
                new[s, i] = m
            elif CY[i] == 1:
                new[s, i, 1:] = m[:-1]
                new[s, OPP[i], -1] = o[-1]
            else:
                new[s, i, :-1] = m[1:]
                new[s, OPP[i], 0] = o[0]
    return new


def _exact_flow(case: dict, seed: int, steps: int) -> torch.Tensor:
    f = _populations(case, seed, case["nx"], case["ny"]).double()
    for _ in range(steps):
        f = _exact_step(f, case)
    return f


def _host(t: torch.Tensor) -> np.ndarray:
    return t.cpu().numpy()


def _dx(a):
    return 0.5 * (torch.roll(a, -1, 1) - torch.roll(a, 1, 1))


def _dy(a):
    """Centred differences along y; the rows beside the ends are never averaged."""
    return 0.5 * (torch.roll(a, -1, 0) - torch.roll(a, 1, 0))


def _stored(f: torch.Tensor, case: dict) -> torch.Tensor:
    """The state the handle holds after it is given f: 16-bit storage rounds
    f - w_i rho0_s, rho0_s the mean of a component's two bulk densities."""
    if case["storage"] != "f32":
        t = torch.float16 if case["storage"] == "f16" else torch.bfloat16
        for s, mass in enumerate((MASS_A, MASS_B)):
            for i in range(9):
                shift = np.float32(W[i]) * np.float32(0.5 * mass * (1 + case["minority"]))
                f[s, i] = (f[s, i] - float(shift)).to(t).float() + float(shift)
    return f.double()


def _exact_diagnostics(case: dict, seed: int) -> dict:
    """The averages of the energy budget over the rows away from the walls."""
    f = _stored(_populations(case, seed, case["nx"], case["ny"]), case)
    nx, ny, g, G = case["nx"], case["ny"], case["g"], case["G"]
    crop = min(CROP, ny // 4)
    A, B = f.sum(1)
    rho, phi = A + B, A - B
    jx, jy = _momenta(f)
    acc = _accelerations(torch.stack([A, B]), case)
    ux, uy = ((j + 0.5 * (A * acc[0][k] + B * acc[1][k])) / rho for k, j in enumerate((jx, jy)))

    def mean(a):
        return float(a[crop:ny - crop].mean())

    def flux(xx, xy, yy):
        return mean(ux * (_dx(xx) + _dy(xy)) + uy * (_dx(xy) + _dy(yy)))

    cs2 = 1.0 / 3.0
    kappa, spurious = cs2 * cs2 * G / 4, cs2 * cs2 * 0.25
    pb = cs2 * rho + G * cs2 / 4 * (rho * rho - phi * phi)
    px, py = _dx(phi), _dy(phi)
    lap = torch.roll(phi, 1, 0) + torch.roll(phi, -1, 0) + torch.roll(phi, 1, 1) + torch.roll(phi, -1, 1) - 4 * phi
    iso = -kappa * phi * lap - 0.5 * kappa * (px * px + py * py)
    vx, vy = B * _dx(A) - A * _dx(B), B * _dy(A) - A * _dy(B)
    k = spurious / (torch.clamp(A * B, min=1e-12) * rho)
    om = _dx(uy) - _dy(ux)
    rho_bar = mean(rho)
    rows = torch.arange(ny, dtype=torch.float64, device="cuda")[:, None]
    eps = case["minority"]
    top, bot = MASS_A / (MASS_A + eps * MASS_B), eps * MASS_A / (eps * MASS_A + MASS_B)
    c = ((A / rho)[crop:ny - crop].mean(1) - bot) / (top - bot)
    c = c.clamp(0.0, 1.0)
    b = phi[crop:ny - crop] > 0
    cc = [int((b != torch.roll(b, -1, 1)).sum())] + [int((b[:-1] != torch.roll(b[1:], d, 1)).sum()) for d in (0, -1, 1)]
    terms = dict(
        mass_A=float(A.sum()), mass_B=float(B.sum()), E_k=mean(0.5 * rho * (ux * ux + uy * uy)), E_p=g * mean(rows * phi),
        buoyancy=g * mean(uy * phi), flux_pb=mean(ux * _dx(pb) + uy * _dy(pb)),
        flux_K=flux(iso + kappa * px * px, kappa * px * py, iso + kappa * py * py),
        flux_tau=flux(k * vx * vx, k * vx * vy, k * vy * vy),
        viscous=rho_bar * cs2 * 0.5 * flux(2 * _dx(ux), _dx(uy) + _dy(ux), 2 * _dy(uy)),
        enstrophy=0.5 * float((om * om)[crop:ny - crop].sum()), rho_bar=rho_bar, h=6.0 * float((c * (1 - c)).sum()),
        L_int=math.pi / 8 * (cc[0] + cc[1] + (cc[2] + cc[3]) / math.sqrt(2.0)))
    return dict(terms=terms, profile=_host(phi[crop:ny - crop].mean(1)))


def _conv(a: torch.Tensor, w: torch.Tensor, b: torch.Tensor) -> torch.Tensor:
    """3x3 cross-correlation of [C, ny, nx], x periodic and zeros beyond the walls."""
    ny, nx = a.shape[1:]
    p = torch.cat([a[:, :, -1:], a, a[:, :, :1]], 2)
    z = torch.zeros_like(p[:, :1])
    p = torch.cat([z, p, z], 1)
    out = b[:, None].expand(-1, ny * nx)
    for k in range(9):
        out = out + w[:, :, k // 3, k % 3] @ p[:, k // 3:k // 3 + ny, k % 3:k % 3 + nx].reshape(a.shape[0], -1)
    return out.reshape(-1, ny, nx)


def _unpack(p: torch.Tensor) -> list[torch.Tensor]:
    """The layers' weights (stored in BF16 in the convolutions) and biases."""
    out, k = [], 0
    for s in CNN_SHAPES:
        n = math.prod(s)
        v = p[k:k + n].reshape(s)
        out.append((v.bfloat16() if len(s) == 4 else v).double())
        k += n
    return out


def _exact_network(p: list[torch.Tensor], x: torch.Tensor) -> torch.Tensor:
    return _conv(torch.relu(_conv(torch.relu(_conv(x, p[0], p[1])), p[2], p[3])), p[4], p[5])


def _exact_correction(f: torch.Tensor, case: dict, net: list[torch.Tensor]) -> torch.Tensor:
    """The closure's interface correction: the order parameter and a quarter of the
    velocity, each component's mass kept, the non-equilibrium part in proportion."""
    rho = f.sum(1)
    rt = rho[0] + rho[1]
    jx, jy = _momenta(f)
    acc = _accelerations(rho, case)
    force = [rho[0] * acc[0][k] + rho[1] * acc[1][k] for k in range(2)]
    v = (rho[0], rho[1], (jx + 0.5 * force[0]) / rt, (jy + 0.5 * force[1]) / rt)
    scale = np.asarray(OUT_SCALE, dtype=np.float32).astype(np.float64)
    mean, inv = (np.asarray(a, dtype=np.float32).astype(np.float64) for a in (IN_MEAN, IN_SCALE))
    y = _exact_network(net, torch.stack([(v[k] - mean[k]) / inv[k] for k in range(4)]))
    d = [y[k] * scale[k] for k in range(4)]
    eps = case["minority"]
    top, bot = MASS_A / (MASS_A + eps * MASS_B), eps * MASS_A / (eps * MASS_A + MASS_B)
    c = ((rho[0] / rt - bot) / (top - bot)).clamp(0.0, 1.0)
    w = 4 * c * (1 - c)
    h = torch.minimum(torch.maximum(0.5 * w * (d[0] - d[1]), -0.5 * rho[0]), 0.5 * rho[1])
    dA = h - w * (h.sum() / w.sum())
    bx, by = jx / rt, jy / rt
    vx, vy = bx + 0.25 * d[2], by + 0.25 * d[3]
    out = torch.empty_like(f)
    for s in range(2):
        r1 = torch.clamp(rho[s] + (dA if s == 0 else -dA), min=0.0)
        q = torch.where(rho[s] > 0, r1 / rho[s], torch.zeros_like(r1))
        for i in range(9):
            out[s, i] = _equilibrium(i, r1, vx, vy) + q * (f[s, i] - _equilibrium(i, rho[s], bx, by))
    return out


def exact(case: dict, seed: int):
    kind = case["kind"]
    if kind == "step":
        if case["nx"] * case["ny"] * case["steps"] > 12e9:   # over 20 s in 64 bits
            return None
        return _host(_exact_flow(case, seed, case["steps"]))
    if kind == "noalloc":
        return _host(_exact_flow(case, seed, 1))
    if kind == "diagnostics":
        return _exact_diagnostics(case, seed)
    if kind == "ensemble":
        return [_host(_exact_flow(m, seed * 100 + i, case["steps"])) for i, m in enumerate(_members(case))]
    net = _unpack(torch.from_numpy(_network(seed)).cuda())
    if kind == "closure":
        f = _exact_flow(case, seed, 0)
        for _ in range(case["intervals"]):
            for _ in range(CLOSURE_INTERVAL):
                f = _exact_step(f, case)
            f = _exact_correction(f, case, net)
        return _host(f)
    x, t = _images(case, seed)
    if kind == "infer":
        return _host(_exact_network(net, x.double()))
    net = [p.requires_grad_() for p in net]
    loss = ((_exact_network(net, x.double()) - t.double()) ** 2).mean()
    loss.backward()
    return dict(loss=float(loss.detach()), grad=_host(torch.cat([p.grad.reshape(-1) for p in net])))
