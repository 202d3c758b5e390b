"""The work that a user of this library has it do, as cases to be timed.

A case is one public call sequence of the library on inputs made from a seed: some
timesteps of a 1D, batched, FP64 or 2D simulation and the read-back of its fields, one
allocation-free particle step, one field solve, one pass of the U-Net.  ``prepare``
makes what a program holds before that (the handle with its particles, the network with
its weights), ``run`` is one pass.

Particles have no defined order after a step, so the simulations' outputs are the nodal
fields and the int64 fixed-point deposits, which depend on every bit of every particle.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1511_08225_gb300 import binding, binding2d, binding_unet, inputs

ONE, HEAVISIDE, RELATIVISTIC = inputs.BETA_ONE, inputs.BETA_HEAVISIDE, inputs.BETA_RELATIVISTIC


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the paper's argon sheath (Sec. IV): 100 cells fed through the right plate, some
        # 10^5 macroparticles; the study that the method is quoted on, hundreds of short
        # steps with a look at the profiles now and then
        {"name": "paper_sheath_100", "path": "sheath1d", "source": "wall", "cells": 100, "ppc": 1000,
         "kind": HEAVISIDE, "v0": 0.016, "profile": False, "settle": 600, "steps": 32},
        # the periodic electron-ion plasma of 256 cells and 51,200 particles
        {"name": "periodic_256", "path": "periodic1d", "cells": 256, "ppc": 100, "kind": HEAVISIDE,
         "v0": 0.2, "steps": 32},
        # the same plasma in the plain FP64 form, which a user checks the mixed form with
        {"name": "fp64_periodic_256", "path": "fp64", "cells": 256, "ppc": 100, "kind": HEAVISIDE,
         "v0": 0.2, "steps": 8},
        # an odd-sized sheath of half a million particles with the smooth (relativistic)
        # beta and a speed limit that varies in space
        {"name": "sheath_1237_profile", "path": "sheath1d", "source": "loss", "cells": 1237, "ppc": 211,
         "kind": RELATIVISTIC, "v0": 0.05, "profile": True, "settle": 1024, "steps": 32},
        # the argon-like sheath that the benchmark runs: 4,096 cells, 8.19M particles, in
        # its saturated state
        {"name": "sheath_4096", "path": "sheath1d", "source": "loss", "cells": 4096, "ppc": 1000,
         "kind": HEAVISIDE, "v0": 0.02, "profile": False, "settle": 2048, "steps": 32},
        # a parameter scan: independent sheaths of uneven size and speed limit in one batch
        {"name": "batch_48", "path": "batch", "members": 48, "cells_lo": 512, "cells_hi": 4096,
         "ppc_lo": 100, "ppc_hi": 500, "scan": inputs.SEED, "settle": 32, "steps": 16},
        # one species stepped on a caller's own arrays, a ragged million particles
        {"name": "noalloc_1m", "path": "noalloc", "cells": 1024, "n": 1000003, "kind": HEAVISIDE,
         "v0": 0.05, "periodic": False},
        # 2D plasma between plates with the direct solver: a small run, short steps
        {"name": "plasma2d_256_fft", "path": "plasma2d", "solver": "fft", "nx": 256, "ny": 256, "ppc": 16,
         "v0": 0.1, "steps": 16},
        # ... and the 1,024 x 1,024 grid
        {"name": "plasma2d_1024_fft", "path": "plasma2d", "solver": "fft", "nx": 1024, "ny": 1024,
         "ppc": 32, "v0": 0.1, "steps": 16},
        # 2D with the default solver (conjugate gradients from the previous potential), on
        # a grid whose width is no power of two
        {"name": "plasma2d_250_cg", "path": "plasma2d", "solver": "cg", "nx": 250, "ny": 241, "ppc": 16,
         "v0": 0.1, "steps": 2},
        # the warm-start network on one charge image of the 1,024 x 1,024 grid (inference)
        {"name": "unet_forward_1024", "path": "unet_forward", "levels": 4, "base": 32, "h": 1024,
         "w": 1024, "batch": 1, "tensor_cores": True},
        # its training: loss and parameter gradients of a mini-batch
        {"name": "unet_gradients_512", "path": "unet_gradients", "levels": 4, "base": 32, "h": 512,
         "w": 512, "batch": 2, "loss": "energy", "tensor_cores": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["wall1d", "loss1d", "loss1d", "periodic1d", "fp64", "batch", "noalloc", "fft2d",
                       "fft2d", "cg2d", "poisson2d", "unet_forward", "unet_forward", "unet_gradients"])
    if path == "wall1d":
        kind = rng.choice([ONE, HEAVISIDE, RELATIVISTIC])
        return {"path": "sheath1d", "source": "wall", "cells": _log_int(rng, 60, 400),
                "ppc": _log_int(rng, 100, 1500), "kind": kind, "v0": round(rng.uniform(0.01, 0.1), 4),
                "profile": False, "settle": 600, "steps": 32}
    if path == "loss1d":
        cells = _log_int(rng, 200, 8192)
        return {"path": "sheath1d", "source": "loss", "cells": cells,
                "ppc": _log_int(rng, 50, min(1000, 4_000_000 // cells)),
                "kind": rng.choice([HEAVISIDE, HEAVISIDE, RELATIVISTIC]),
                "v0": round(math.exp(rng.uniform(math.log(0.01), math.log(0.5))), 4),
                "profile": rng.random() < 0.25, "settle": 1024, "steps": 32}
    if path in ("periodic1d", "fp64"):
        cells = _log_int(rng, 64, 2048)
        return {"path": path, "cells": cells,
                "ppc": _log_int(rng, 20, min(1000, (2_000_000 if path == "periodic1d" else 300_000) // cells)),
                "kind": rng.choice([ONE, HEAVISIDE, RELATIVISTIC]), "v0": round(rng.uniform(0.1, 0.5), 3),
                "steps": 32 if path == "periodic1d" else 8}
    if path == "batch":
        lo = _log_int(rng, 64, 1024)
        return {"path": "batch", "members": _log_int(rng, 2, 64), "cells_lo": lo, "cells_hi": 4 * lo,
                "ppc_lo": 100, "ppc_hi": _log_int(rng, 150, 500), "scan": rng.randrange(1 << 30),
                "settle": 32, "steps": 16}
    if path == "noalloc":
        return {"path": "noalloc", "cells": _log_int(rng, 64, 16000), "n": _log_int(rng, 1000, 8_000_000),
                "kind": rng.choice([ONE, HEAVISIDE, RELATIVISTIC]), "v0": round(rng.uniform(0.01, 0.3), 4),
                "periodic": rng.random() < 0.5}
    if path == "fft2d":
        nx, ny = 1 << rng.randint(6, 10), _log_int(rng, 33, 1024)
        return {"path": "plasma2d", "solver": "fft", "nx": nx, "ny": ny,
                "ppc": _log_int(rng, 4, min(64, max(5, 30_000_000 // (nx * ny)))),
                "v0": round(rng.uniform(0.05, 0.3), 3), "steps": 16}
    if path == "cg2d":
        return {"path": "plasma2d", "solver": "cg", "nx": _log_int(rng, 48, 512), "ny": _log_int(rng, 48, 512),
                "ppc": _log_int(rng, 4, 32), "v0": round(rng.uniform(0.05, 0.3), 3), "steps": 1}
    if path == "poisson2d":
        return {"path": "poisson2d", "solver": rng.choice(["cg", "fft"]), "nx": 1 << rng.randint(6, 10),
                "ny": _log_int(rng, 48, 1024)}
    levels = rng.randint(2, 4)
    step = 1 << (levels - 1)
    top = 1024 if path == "unet_forward" else 512
    tc = rng.random() < 0.8
    hi = top if tc else 192
    case = {"path": path, "levels": levels, "base": rng.choice([8, 16, 32]),
            "h": step * _log_int(rng, 40 // step, hi // step), "w": step * _log_int(rng, 40 // step, hi // step),
            "batch": rng.randint(1, 2 if path == "unet_forward" else 3), "tensor_cores": tc}
    if path == "unet_gradients":
        case["loss"] = rng.choice(["mse", "energy"])
    return case


# ------------------------------------------------------------------ inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _g_velocities(g, n, vth, v0, kind):
    """n velocities of the speed-limited load g0 = f0 / beta, f0 a Maxwellian (vth per
    component): rejection from the Maxwellian times (1 + r/v0), float32 on the GPU."""
    out = torch.randn((n, 3), generator=g, device="cuda").mul_(vth)
    if kind == ONE:
        return out
    mean_r = vth * 2.0 * math.sqrt(2.0 / math.pi)
    weighted = (mean_r / v0) / (1.0 + mean_r / v0)
    filled = 0
    while filled < n:
        m = int(1.5 * (n - filled)) + 1024
        u = torch.rand((4, m), generator=g, device="cuda")
        plain = torch.randn((m, 3), generator=g, device="cuda").square_().sum(1).sqrt_()
        gamma2 = -(torch.log(1.0 - u[1]) + torch.log(1.0 - u[2]))
        r = vth * torch.where(u[0] < weighted, torch.sqrt(2.0 * gamma2), plain)
        factor = torch.clamp(r / v0, min=1.0) if kind == HEAVISIDE else torch.sqrt(r * r + v0 * v0) / v0
        r = r[u[3] * (1.0 + r / v0) <= factor][:n - filled]
        d = torch.randn((r.numel(), 3), generator=g, device="cuda")
        out[filled:filled + r.numel()] = r[:, None] * d / d.norm(dim=1, keepdim=True)
        filled += r.numel()
    return out


def _load_1d(g, prob, h, instance=0):
    n_cells = prob["n_cells"]
    for s, sp in enumerate(prob["species"]):
        n = sp["ppc"] * n_cells
        cell = torch.randint(0, n_cells, (n,), generator=g, device="cuda", dtype=torch.int32)
        off = torch.rand((n,), generator=g, device="cuda")
        v = _g_velocities(g, n, sp["vth"], sp["v0"], sp["kind"])
        torch.cuda.synchronize()  # the handle works on its own stream
        binding.slpic_load_particles_dev(h, instance, s, cell, off, v)


def _sheath_problem(case, seed):
    if case["source"] == "wall":
        prob = inputs.paper_sheath_problem(kind=case["kind"], n_cells=case["cells"], v0=case["v0"],
                                           ppc=case["ppc"], seed=seed)
    else:
        prob = inputs.sheath_problem(n_cells=case["cells"], ppc=case["ppc"], v0=case["v0"], kind=case["kind"],
                                     seed=seed, capacity_factor=_CAPACITY)
    if case["profile"]:  # half the limit at the plates, the full one in the middle
        x = (np.arange(case["cells"]) + 0.5) / case["cells"]
        prob["v0_profile"] = 0.5 + 0.5 * np.sin(np.pi * x)
    return prob


def _unet_params(case, seed):
    """He-normal weights and small biases, (W, b) per conv in parameter order."""
    rng = np.random.default_rng(seed)
    ch = [case["base"] << l for l in range(case["levels"])]
    shapes = [(1, ch[0])] + [(ch[l - 1], ch[l]) for l in range(1, len(ch))]
    shapes += [(ch[l + 1] + ch[l], ch[l]) for l in range(len(ch) - 2, -1, -1)] + [(ch[0], 1)]
    return [(rng.normal(0.0, math.sqrt(2.0 / (9.0 * ci)), (co, ci, 3, 3)).astype(np.float32),
             rng.normal(0.0, 0.05, co).astype(np.float32)) for ci, co in shapes]


def _unet_images(case, seed):
    """Charge images (shot noise on a smooth part, the plate row zero) and potential-like
    targets (their Poisson images on a periodic box)."""
    g = _generator(seed)
    nb, h, w = case["batch"], case["h"], case["w"]
    x = torch.randn((nb, h, w), generator=g, device="cuda")
    y = torch.arange(h, device="cuda")[:, None] / h
    x = x + 0.5 * torch.sin(2 * math.pi * y) * torch.rand((nb, 1, 1), generator=g, device="cuda")
    x[:, 0] = 0.0
    kx = 2.0 - 2.0 * torch.cos(2 * math.pi * torch.arange(w // 2 + 1, device="cuda") / w)
    ky = 2.0 - 2.0 * torch.cos(2 * math.pi * torch.arange(h, device="cuda") / h)
    k2 = kx[None, :] + ky[:, None]
    k2[0, 0] = 1.0
    t = torch.fft.irfft2(torch.fft.rfft2(x - x.mean((1, 2), keepdim=True)) / k2, s=(h, w))
    t[:, 0] = 0.0
    return x.contiguous(), t.contiguous()


_OUT_SCALE = 4.0  # the network's output factor: about rms(potential) / rms(charge)


def _noalloc_inputs(case, seed):
    g = _generator(seed)
    n, cells = case["n"], case["cells"]
    cell = torch.randint(0, cells, (n,), generator=g, device="cuda", dtype=torch.int32)
    state = torch.empty((n, 4), device="cuda")
    state[:, 0] = torch.rand((n,), generator=g, device="cuda")
    state[:, 1:] = _g_velocities(g, n, 1.0, case["v0"], case["kind"])
    nodes = cells + (0 if case["periodic"] else 1)
    x = torch.arange(nodes, device="cuda") / cells
    field = 0.05 * torch.sin(2 * math.pi * x) + 0.01 * torch.randn((nodes,), generator=g, device="cuda")
    return cell, state, field


def _poisson_rho(case, seed):
    rng = np.random.default_rng(seed)
    y = np.arange(case["ny"] + 1)[:, None] / case["ny"]
    return 0.1 * np.sin(np.pi * y) + 0.2 * rng.normal(size=(case["ny"] + 1, case["nx"]))


# Slots per loaded particle: a long run's source fills the slots of absorbed particles
# only at the compacting steps, so it is given more than the generators' default.
_CAPACITY = 3.0


# ------------------------------------------------------------------ prepare
def prepare(case, seed):
    path, seed = case["path"], int(seed)
    if path == "sheath1d":
        prob = _sheath_problem(case, seed)
        sim = binding.Simulation(prob)
        if case["source"] == "loss":  # the wall-fed sheath starts empty and fills
            _load_1d(_generator(seed), prob, sim.h)
        sim.prepare()
        sim.step(case["settle"])
        sim.synchronize()
        return {"path": path, "sim": sim, "steps": case["steps"]}
    if path == "periodic1d":
        prob = inputs.periodic_problem(n_cells=case["cells"], ppc=case["ppc"], v0=case["v0"], kind=case["kind"],
                                       seed=seed)
        sim = binding.Simulation(prob)
        _load_1d(_generator(seed), prob, sim.h)
        sim.prepare()
        sim.synchronize()
        return {"path": path, "sim": sim, "steps": case["steps"]}
    if path == "fp64":
        prob = inputs.periodic_problem(n_cells=case["cells"], ppc=case["ppc"], v0=case["v0"], kind=case["kind"],
                                       seed=seed)
        sim, g = binding.SimulationFP64(prob), _generator(seed)
        for s, sp in enumerate(prob["species"]):
            n = sp["ppc"] * prob["n_cells"]
            x = torch.rand((n,), generator=g, device="cuda", dtype=torch.float64) * (prob["n_cells"] * prob["dx"])
            v = _g_velocities(g, n, sp["vth"], sp["v0"], sp["kind"]).double()
            sim.load(s, x.cpu().numpy(), v.cpu().numpy())
        sim.prepare()
        sim.synchronize()
        return {"path": path, "sim": sim, "steps": case["steps"]}
    if path == "batch":
        # the scan's sizes and speed limits belong to the case, particles and source to the seed
        probs = inputs.batch_problems(m=case["members"], seed=case["scan"],
                                      cells=(case["cells_lo"], case["cells_hi"]),
                                      ppc=(case["ppc_lo"], case["ppc_hi"]))
        for i, prob in enumerate(probs):
            prob["seed"] = seed + i
            for sp in prob["species"]:
                sp["capacity"] = int(_CAPACITY * sp["ppc"] * prob["n_cells"]) + 1024
        sim, g = binding.Batch(probs), _generator(seed)
        for i, prob in enumerate(probs):
            _load_1d(g, prob, sim.h, i)
        sim.prepare()
        sim.step(case["settle"])
        sim.synchronize()
        return {"path": path, "sim": sim, "steps": case["steps"]}
    if path == "noalloc":
        prob = inputs.periodic_problem(n_cells=case["cells"], dt=0.5 / case["v0"], v0=case["v0"],
                                       kind=case["kind"], seed=seed)
        if case["kind"] == ONE:
            prob["dt"] = 0.1
        prob["periodic"] = case["periodic"]
        cell, state, field = _noalloc_inputs(case, seed)
        return {"path": path, "cfg": binding.config_from_problem(prob), "cell": cell, "state": state,
                "E": field, "cell_out": torch.empty_like(cell), "state_out": torch.empty_like(state),
                "charge": torch.empty(field.numel(), dtype=torch.int64, device="cuda")}
    if path == "plasma2d":
        prob = inputs.plasma2d_problem(nx=case["nx"], ny=case["ny"], ppc=case["ppc"], v0=case["v0"],
                                       solver=case["solver"], seed=seed, capacity_factor=_CAPACITY)
        sim, g = binding2d.Simulation2D(prob), _generator(seed)
        for s, sp in enumerate(prob["species"]):
            n = case["ppc"] * case["nx"] * case["ny"]
            cell = torch.randint(0, case["nx"] * case["ny"], (n,), generator=g, device="cuda", dtype=torch.int32)
            off = torch.rand((n, 2), generator=g, device="cuda")
            v = _g_velocities(g, n, sp["vth"], sp["v0"], sp["kind"])
            sim.load(s, cell.cpu().numpy(), off.cpu().numpy(), v.cpu().numpy())
        sim.prepare()
        sim.synchronize()
        return {"path": path, "sim": sim, "steps": case["steps"]}
    if path == "poisson2d":
        prob = inputs.plasma2d_problem(nx=case["nx"], ny=case["ny"], ppc=1, solver=case["solver"], seed=seed)
        return {"path": path, "sim": binding2d.Simulation2D(prob), "rho": _poisson_rho(case, seed)}
    net = binding_unet.UNet(case["levels"], case["base"], case["h"], case["w"], max_batch=case["batch"],
                            normalise=True, out_scale=_OUT_SCALE, tensor_cores=case["tensor_cores"],
                            loss=(binding_unet.SLPIC_UNET_LOSS_ENERGY if case.get("loss") == "energy"
                                  else binding_unet.SLPIC_UNET_LOSS_MSE))
    net.set_params(_unet_params(case, seed))
    x, t = _unet_images(case, seed)
    return {"path": path, "net": net, "x": x, "t": t, "y": torch.empty_like(x)}


# ------------------------------------------------------------------ run
def run(state):
    path = state["path"]
    if path in ("sheath1d", "periodic1d"):
        sim = state["sim"]
        sim.step(state["steps"])
        rho, phi, field = sim.fields()
        return {"rho": rho, "phi": phi, "E": field, "charge": [sim.charge_raw(s) for s in range(sim.ns)]}
    if path == "fp64":
        sim = state["sim"]
        sim.step(state["steps"])
        rho, phi, field = sim.fields()
        return {"rho": rho, "phi": phi, "E": field}
    if path == "batch":
        sim = state["sim"]
        sim.step(state["steps"])
        each = [sim.fields(i) for i in range(len(sim.probs))]
        return {k: np.concatenate([f[j] for f in each]) for j, k in enumerate(("rho", "phi", "E"))}
    if path == "noalloc":
        n_out, absorbed = binding.slpic_particle_step_noalloc(
            state["cfg"], 0, state["cell"], state["state"], state["E"], state["cell_out"], state["state_out"],
            state["charge"], stream=torch.cuda.current_stream().cuda_stream)
        return {"charge": state["charge"], "n_out": n_out, "absorbed": absorbed}
    if path == "plasma2d":
        sim = state["sim"]
        sim.step(state["steps"])
        rho, phi, ex, ey = sim.fields()
        return {"rho": rho, "phi": phi, "Ex": ex, "Ey": ey}
    if path == "poisson2d":
        return {"phi": state["sim"].solve_poisson(state["rho"])[0]}
    if path == "unet_forward":
        state["net"].forward(state["x"], state["y"])
        return {"y": state["y"]}
    loss, grads = state["net"].gradients(state["x"], state["t"])
    return {"loss": loss, "grads": grads}


# ------------------------------------------------------------------ work and exact values
def _conv_macs(case):
    L, C, hw = case["levels"], case["base"], case["h"] * case["w"]
    ch = [C << l for l in range(L)]
    macs = hw * 9 * (ch[0] + ch[0])
    macs += sum(hw // 4 ** l * 9 * ch[l - 1] * ch[l] for l in range(1, L))
    macs += sum(hw // 4 ** l * 9 * (ch[l + 1] + ch[l]) * ch[l] for l in range(L - 1))
    return macs * case["batch"]


def work(case):
    """State read and written once per step (20 bytes a particle in 1D, 24 in 2D, 32 in
    FP64, each way), images and grids once; some 60 flops a particle and step in 1D."""
    path = case["path"]
    if path in ("sheath1d", "periodic1d", "fp64"):
        n = 2 * case["cells"] * case["ppc"] * case["steps"]
        return {"bytes": (64 if path == "fp64" else 40) * n, "flops": 60 * n}
    if path == "batch":
        n = (case["members"] * (case["cells_lo"] + case["cells_hi"]) * (case["ppc_lo"] + case["ppc_hi"]) / 2
             * case["steps"])
        return {"bytes": 40 * n, "flops": 60 * n}
    if path == "noalloc":
        return {"bytes": 40 * case["n"] + 12 * case["cells"], "flops": 60 * case["n"]}
    if path == "plasma2d":
        n = 2 * case["nx"] * case["ny"] * case["ppc"] * case["steps"]
        grid = case["nx"] * case["ny"] * case["steps"]
        return {"bytes": 48 * n + 40 * grid, "flops": 120 * n}
    if path == "poisson2d":
        n = case["nx"] * case["ny"]
        return {"bytes": 16 * n, "flops": 20 * n * math.log2(case["nx"])}
    pixels = case["batch"] * case["h"] * case["w"]
    macs = _conv_macs(case)
    if path == "unet_forward":
        return {"bytes": 8 * pixels, "flops": 2 * macs}
    return {"bytes": 8 * pixels, "flops": 6 * macs}


def _exact_unet(case, seed, gradients):
    """The network in FP64 on the BF16 copies of the weights, activations not rounded."""
    F = torch.nn.functional
    params = [(torch.tensor(w, device="cuda").bfloat16().double().requires_grad_(gradients),
               torch.tensor(b, device="cuda").double().requires_grad_(gradients))
              for w, b in _unet_params(case, seed)]
    x, t = (v.double()[:, None] for v in _unet_images(case, seed))
    s = x.square().mean((2, 3), keepdim=True).sqrt()
    L = case["levels"]
    enc, a = [], x / s
    for l in range(L):
        a = F.relu(F.conv2d(F.avg_pool2d(a, 2) if l else a, *params[l], padding=1))
        enc.append(a)
    for k, l in enumerate(range(L - 2, -1, -1)):
        up = a.repeat_interleave(2, 2).repeat_interleave(2, 3)
        a = F.relu(F.conv2d(torch.cat([up, enc[l]], 1), *params[L + k], padding=1))
    y = F.conv2d(a, *params[-1], padding=1)
    if not gradients:
        return {"y": (y * s * _OUT_SCALE)[:, 0].float().double()}
    e = y - t / (s * _OUT_SCALE)
    if case["loss"] == "energy":
        e = torch.cat([torch.zeros_like(e[:, :, :1]), e[:, :, 1:]], 2)
        dy = F.pad(e, (0, 0, 1, 1))
        ae = 4 * e - e.roll(1, 3) - e.roll(-1, 3) - dy[:, :, :-2] - dy[:, :, 2:]
        loss = (e[:, :, 1:] * ae[:, :, 1:]).sum() / e.numel()
    else:
        loss = e.square().mean()
    flat = torch.autograd.grad(loss, [p for wb in params for p in wb])
    return {"loss": float(loss.detach()),
            "grads": [[flat[2 * k], flat[2 * k + 1]] for k in range(len(params))]}


def exact(case, seed):
    path = case["path"]
    if path == "poisson2d":
        nx, ny = case["nx"], case["ny"]
        b = np.fft.fft(_poisson_rho(case, seed)[1:ny], axis=1)  # dx = eps0 = 1, plates at 0
        diag = (4.0 - 2.0 * np.cos(2 * np.pi * np.arange(nx) / nx))[None, :]
        c = np.zeros((ny - 1, nx))
        d = np.zeros((ny - 1, nx), complex)
        c[0], d[0] = 1.0 / diag, b[0] / diag[0]
        for j in range(1, ny - 1):
            m = 1.0 / (diag[0] - c[j - 1])
            c[j], d[j] = m, (b[j] + d[j - 1]) * m
        for j in range(ny - 3, -1, -1):
            d[j] += c[j] * d[j + 1]
        phi = np.zeros((ny + 1, nx))
        phi[1:ny] = np.fft.ifft(d, axis=1).real
        return {"phi": phi}
    if path in ("unet_forward", "unet_gradients"):
        return _exact_unet(case, seed, path == "unet_gradients")
    return None  # a whole simulation, or integers
