"""The workloads this framework's speed is measured on, through its public entry points.

A case is a dict of plain values; `kind` says which entry points it goes through:

step      One run of the plasma: `Simulation.step(n)`, then what a run reads between two bursts of
          steps: the moments and the potential (on the device), and on the small grids every particle.
          The prepared state has run past the transient in which the preloaded electrons leave, so the
          sources keep its population steady.
ensemble  The same for several independent runs of uneven sizes in one handle.
coupled   A surface model in the loop: every step uploads the electrons it emits, steps once and reads
          the ions that hit the cathode; variable weights, charge exchange and the external circuit on.
solve     `Simulation.solve`: the field of a given charge density, on host arrays.
static    `pic_poisson_solve_static`: the same on device buffers, for callers that cannot allocate.
forward   The network of the learned warm start: one inference.
gradient  The same network's training pass: forward, backward, weight gradients.

The mixed store keeps particles and fields in 32 bits and solves to a relative residual of 1e-8, so its
numbers are returned as 32-bit ones, the counters of events among them: a draw at the edge of a decision
falls either way between two runs, whose deposits sum in another order. The FP64 store is the reference path and is run as the parity tests
run it, solved to 1e-13; its numbers are 64-bit ones. Iteration counts and residuals of the solves say how
a result was reached and are no part of it.
"""
import math

import numpy as np
import torch

import paper_2606_05893_gb300 as pic
from paper_2606_05893_gb300 import workloads as W

FIELD = 9.375e9  # V/m, the applied field of the at-scale workload
RTOL = {"mixed": 1e-8, "fp64": 1e-13}


def listed():
    return [
        # the smallest runs: the paper-sized box with 1e4 superparticles, where latency and launches count
        {"name": "step_mixed_32x32x64", "kind": "step", "precision": "mixed", "nx": 32, "ny": 32, "nz": 64,
         "particles": 10_000, "steps": 20, "read_particles": True},
        {"name": "step_fp64_32x32x64", "kind": "step", "precision": "fp64", "nx": 32, "ny": 32, "nz": 64,
         "particles": 10_000, "steps": 20, "read_particles": True},
        # the at-scale workload (the benchmark's own): production runs
        {"name": "step_mixed_128x128x256", "kind": "step", "precision": "mixed", "nx": 128, "ny": 128, "nz": 256,
         "particles": 10_000_000, "steps": 5, "read_particles": False},
        # the FP64 store at the size of the mixed path's error subcase
        {"name": "step_fp64_64x64x128", "kind": "step", "precision": "fp64", "nx": 64, "ny": 64, "nz": 128,
         "particles": 781_250, "steps": 5, "read_particles": False},
        # the finest grid the benchmark runs
        {"name": "step_mixed_256x256x512", "kind": "step", "precision": "mixed", "nx": 256, "ny": 256, "nz": 512,
         "particles": 20_000_000, "steps": 2, "read_particles": False},
        # a parameter scan: independent runs of uneven sizes side by side
        {"name": "ensemble_mixed_8", "kind": "ensemble", "instances": 8, "mix": 3, "steps": 10},
        # a surface model in the loop, on a box that fits the emitter and no power of two
        {"name": "coupled_40x36x90", "kind": "coupled", "nx": 40, "ny": 36, "nz": 90, "particles": 200_000, "steps": 5,
         "emitted": 256},
        # a field for a density computed elsewhere, on the host, and on device memory that the caller owns
        {"name": "solve_fp64_96x80x150", "kind": "solve", "nx": 96, "ny": 80, "nz": 150},
        {"name": "static_64x64x64", "kind": "static", "nx": 64, "ny": 64, "nz": 64},
        # the learned warm start: inference on the at-scale grid, a training pass on the test grid
        {"name": "forward_256x128x128", "kind": "forward", "D": 256, "H": 128, "W": 128},
        {"name": "gradient_64x32x32", "kind": "gradient", "D": 64, "H": 32, "W": 32},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "ensemble", "coupled", "solve", "static", "forward", "gradient"])
    if kind == "step":
        precision = rng.choice(["mixed", "mixed", "fp64"])
        top = 160 if precision == "mixed" else 96
        n = 4 * _log_int(rng, 6, top // 4)
        ny = n if rng.random() < 0.6 else 4 * _log_int(rng, 6, top // 4)
        nz = 2 * _log_int(rng, n // 2, 3 * n // 2)
        cells = n * ny * nz
        particles = min(_log_int(rng, 10_000, 10_000_000 if precision == "mixed" else 1_000_000), 4 * cells)
        small = particles <= 50_000
        return {"kind": "step", "precision": precision, "nx": n, "ny": ny, "nz": nz, "particles": particles,
                "steps": 20 if small else 5, "read_particles": small}
    if kind == "ensemble":
        return {"kind": "ensemble", "instances": rng.randint(3, 8), "mix": rng.randint(4, 1_000_000), "steps": 10}
    if kind == "coupled":
        nx, ny = 2 * _log_int(rng, 12, 32), 2 * _log_int(rng, 12, 32)
        return {"kind": "coupled", "nx": nx, "ny": ny, "nz": _log_int(rng, 40, 130), "particles": _log_int(rng, 20_000, 400_000),
                "steps": 5, "emitted": _log_int(rng, 32, 1024)}
    if kind == "solve":
        return {"kind": "solve", "nx": 2 * _log_int(rng, 8, 64), "ny": 2 * _log_int(rng, 8, 64), "nz": _log_int(rng, 24, 256)}
    if kind == "static":
        nx, ny = _log_int(rng, 12, 64), _log_int(rng, 12, 64)
        return {"kind": "static", "nx": nx, "ny": ny, "nz": min(_log_int(rng, 24, 128), 1 + pic.PIC_STATIC_MAX_UNKNOWNS // (nx * ny))}
    if kind == "forward":
        side = 8 * rng.randint(4, 16)
        return {"kind": "forward", "D": 8 * rng.randint(4, 32), "H": side, "W": side if rng.random() < 0.7 else 8 * rng.randint(4, 16)}
    return {"kind": "gradient", "D": 8 * rng.randint(2, 12), "H": 8 * rng.randint(2, 8), "W": 8 * rng.randint(2, 8)}


# ---------------------------------------------------------------------------
# the plasma: the at-scale workload's physics on any box, its preload made on the GPU
# ---------------------------------------------------------------------------
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _plasma(nx, ny, nz, particles, seed, precision, h=2.5e-9, sort_interval=20):
    """The workload of `config_scale` on an nx x ny x nz box with a preload of `particles`: 60 % electrons in
    a cylinder above the emitter, 30 % Cu and 10 % Cu+ in a cloud over it."""
    Lx, Ly, Lz = nx * h, ny * h, nz * h
    R = min(40e-9, 0.3 * min(Lx, Ly))
    ne, nn = int(round(0.6 * particles)), int(round(0.3 * particles))
    ni = particles - ne - nn
    weight = 0.1 * FIELD * W.EPS0 * Lx * Ly / (W.E_CHARGE * (ne - ni))
    wl = W.config_scale(seed=seed, n_preload=0, nx=nx, ny=ny, nz=nz, h=h, r_emit=R, weight=weight)
    wl.sort_interval, wl.cg_rtol, wl.cg_maxit = sort_interval, RTOL[precision], 4000
    g = _generator(seed)

    def normal(n, T, m):
        return torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float64) * math.sqrt(W.K_B * T / m)

    def uniform(n):
        return torch.rand(n, generator=g, device="cuda", dtype=torch.float64)

    r, th, z = R * uniform(ne).sqrt(), 2 * math.pi * uniform(ne), uniform(ne) * Lz
    x = torch.stack([Lx / 2 + r * th.cos(), Ly / 2 + r * th.sin(), z], 1)
    v = normal(ne, 0.5 * W.E_CHARGE / W.K_B, W.M_E)
    v[:, 2] += (2 * W.E_CHARGE * FIELD / W.M_E * z).sqrt()
    pre = [(x, v)]
    for n in (nn, ni):
        x = torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float64) * torch.tensor([R, R, 2 * R], device="cuda", dtype=torch.float64)
        x[:, 0] += Lx / 2
        x[:, 1] += Ly / 2
        x[:, 2].abs_()
        L = torch.tensor([Lx, Ly, Lz], device="cuda", dtype=torch.float64)
        x = torch.remainder(x, L)
        pre.append((torch.where(x >= L, torch.zeros_like(x), x), normal(n, 2000.0, W.M_CU)))
    wl.preload = [(a.cpu().numpy(), b.cpu().numpy()) for a, b in pre]
    per_step = [s.flux_m2s * math.pi * s.radius ** 2 * wl.dt / weight for s in wl.sources]
    crossing = math.sqrt(2 * W.M_E * Lz / (W.E_CHARGE * FIELD)) / wl.dt  # steps an electron needs to the anode
    for s, sp in enumerate(wl.species):
        sp.capacity = int(1.5 * max(ne, nn, ni) + 3 * crossing * per_step[0] + 20_000 * per_step[1] + 65536)
    return wl, int(1.2 * crossing) + 2


_PRECISION = {"mixed": pic.PIC_MIXED, "fp64": pic.PIC_FP64}


def _moments(m, real):
    """The moments a run records, energies in the store's precision, counters as the store can repeat them."""
    whole = [m["step"], *m["count"], *m["injected"], *m["abs_cathode"], *m["abs_anode"], m["n_ionization"], m["n_elastic"],
             m["n_suppressed"], m["n_cx"], m["next_pid"], *m["pushed"]]
    return {"counts": np.array(whole, dtype=np.int64 if real is np.float64 else real), "kinetic": np.array(m["kinetic"], dtype=real),
            "absorbed_energy": np.array(m["abs_energy_cathode"] + m["abs_energy_anode"], dtype=real),
            "field_energy": np.array([m["field_energy"]], dtype=real), "charge": np.array([m["total_charge"]], dtype=real),
            "anode_V": np.array([m["anode_V"]], dtype=real)}


def _potential(sim, inst, buffer, real):
    pic.pic_get_phi_device(sim.h, inst, buffer.data_ptr())
    return buffer.to(real, copy=True)


def _rows(a, n, dtype, fill=0):
    """`a` as the first rows of an array of n: what a run leaves varies in number, a record of it does not."""
    out = np.full((n, *a.shape[1:]), fill, dtype=dtype)
    out[:min(n, a.shape[0])] = a[:n]
    return out


def _particles(sim, real, n):
    """Every particle, by its identifier (the order of the store is not part of the result)."""
    out = []
    for s in range(3):
        x, v, pid = sim.particles(s)
        order = np.argsort(pid)
        out.append({"pid": _rows(pid[order], n, np.int64, -1), "x": _rows(x[order], n, real), "v": _rows(v[order], n, real)})
    return out


def _nodes(wl):
    return torch.empty((wl.nz + 1, wl.ny, wl.nx), dtype=torch.float64, device="cuda")


def _prepare_step(case, seed):
    wl, settle = _plasma(case["nx"], case["ny"], case["nz"], case["particles"], seed, case["precision"])
    sim = pic.Simulation(wl, precision=_PRECISION[case["precision"]])
    wl.preload = None
    sim.step(settle)
    return {"case": case, "sim": sim, "phi": _nodes(wl)}


def _run_step(s):
    case, sim = s["case"], s["sim"]
    host, dev = (np.float32, torch.float32) if case["precision"] == "mixed" else (np.float64, torch.float64)
    sim.step(case["steps"])
    out = {"moments": _moments(sim.moments(), host), "phi": _potential(sim, 0, s["phi"], dev)}
    if case["read_particles"]:
        out["particles"] = _particles(sim, host, case["particles"])
    return out


def _members(case):
    """Sizes of the ensemble's runs: grids (n, n, 2n) and preloads as the benchmark's ensemble draws them."""
    import random
    rng = random.Random(case["mix"])
    out = []
    for _ in range(case["instances"]):
        n = rng.choice((32, 64, 96, 128))
        out.append((n, n, 2 * n, _log_int(rng, 10_000, 2_000_000)))
    return out


def _prepare_ensemble(case, seed):
    wls, settle = [], 0
    for i, (nx, ny, nz, particles) in enumerate(_members(case)):
        wl, n = _plasma(nx, ny, nz, particles, seed * 64 + i, "mixed", sort_interval=40)
        wls.append(wl)
        settle = max(settle, n)
    sim = pic.Simulation(wls, precision=pic.PIC_MIXED)
    for wl in wls:
        wl.preload = None
    sim.step(settle)
    return {"case": case, "sim": sim, "phi": [_nodes(wl) for wl in wls]}


def _run_ensemble(s):
    sim = s["sim"]
    sim.step(s["case"]["steps"])
    return [{"counts": _moments(sim.moments(i), np.float32)["counts"], "phi": _potential(sim, i, phi, torch.float32)}
            for i, phi in enumerate(s["phi"])]


def _prepare_coupled(case, seed):
    wl, settle = _plasma(case["nx"], case["ny"], case["nz"], case["particles"], seed, "mixed")
    wl.variable_weights = True
    rng = np.random.default_rng(seed)
    wl.preload = [(x, v, rng.integers(1, 5, x.shape[0]).astype(np.uint32)) for x, v in wl.preload]
    wl.xsec = wl.xsec + [W.XSec(W.XS_CHARGE_EXCHANGE, 2, 1, 1, 0.0, np.array([1.0]), np.array([1e-18]))]
    src = wl.sources.pop(0)  # the surface model emits the electrons
    for sp in wl.species:
        sp.capacity += 200 * case["emitted"]
    sim = pic.Simulation(wl, precision=pic.PIC_MIXED)
    wl.preload = None
    pic.pic_set_hit_log(sim.h, 0, 1 << 16)
    pic.pic_set_circuit(sim.h, 0, 1e3, 1e-12, wl.phi_anode)
    batches = []
    for _ in range(16):
        n = case["emitted"]
        r, th = src.radius * np.sqrt(rng.random(n)), 2 * math.pi * rng.random(n)
        x = np.stack([src.cx + r * np.cos(th), src.cy + r * np.sin(th), rng.random(n) * 0.1 * wl.h], axis=1)
        v = rng.standard_normal((n, 3)) * math.sqrt(W.K_B * src.T_K / W.M_E)
        v[:, 2] = np.abs(v[:, 2])
        batches.append((x, v, rng.integers(1, 5, n).astype(np.uint32)))
    s = {"case": case, "sim": sim, "phi": _nodes(wl), "batches": batches, "at": 0}
    for _ in range(settle):
        _coupled_step(s)
    return s


def _coupled_step(s):
    sim = s["sim"]
    pic.pic_inject_particles_m(sim.h, 0, 0, *s["batches"][s["at"] % len(s["batches"])])
    s["at"] += 1
    sim.step(1)
    return pic.pic_get_hits(sim.h, 0)


def _run_coupled(s):
    hits = [_coupled_step(s) for _ in range(s["case"]["steps"])]

    def hit(key, dtype, fill=0):
        return _rows(np.concatenate([h[key] for h in hits]), 4096, dtype, fill)

    return {"hit_pid": hit("pid", np.int64, -1), "hit_step": hit("step", np.int64), "hit_x": hit("x", np.float32),
            "hit_v": hit("v", np.float32), "hit_eV": hit("ke_eV", np.float32),
            "moments": _moments(s["sim"].moments(), np.float32), "phi": _potential(s["sim"], 0, s["phi"], torch.float32)}


# ---------------------------------------------------------------------------
# the field alone
# ---------------------------------------------------------------------------
def _density(nx, ny, nz, seed, h):
    """A charge density as a plasma leaves it: a column over the emitter, graininess of the particles, and a
    net charge that changes the applied field by some ten per cent."""
    g = _generator(seed)
    f64 = {"dtype": torch.float64, "device": "cuda"}
    z, y, x = torch.meshgrid(torch.arange(nz + 1, **f64) / nz, (torch.arange(ny, **f64) - ny / 2) / ny,
                             (torch.arange(nx, **f64) - nx / 2) / nx, indexing="ij")
    shape = torch.exp(-(x * x + y * y) / 0.08) * (0.3 + torch.exp(-4 * z))
    grain = torch.randn(shape.shape, generator=g, **f64)
    scale = 0.2 * FIELD * W.EPS0 / (nz * h)
    return scale * shape * (0.5 + torch.rand(1, generator=g, **f64) + 0.7 * grain)


def _bare(case):
    h = 2.5e-9
    species = W.cu_plasma_species(1.0, 1024)
    return W.Workload("field", case["nx"], case["ny"], case["nz"], h, 0.5e-15, -2.0, FIELD * case["nz"] * h, species, [], [], 1,
                      cg_rtol=1e-13, cg_maxit=20000)


def _prepare_solve(case, seed):
    wl = _bare(case)
    sim = pic.Simulation(wl, precision=pic.PIC_FP64, preload=False)
    return {"case": case, "sim": sim, "rho": _density(wl.nx, wl.ny, wl.nz, seed, wl.h).cpu().numpy()}


def _prepare_static(case, seed):
    wl = _bare(case)
    rho = _density(wl.nx, wl.ny, wl.nz, seed, wl.h)
    return {"case": case, "wl": wl, "rho": rho, "phi": torch.empty_like(rho)}


def _run_static(s):
    wl, phi = s["wl"], s["phi"]
    phi.zero_()
    status, _, _ = pic.pic_poisson_solve_static(wl.nx, wl.ny, wl.nz, wl.h, wl.phi_cathode, wl.phi_anode, s["rho"].data_ptr(),
                                                phi.data_ptr(), 1e-12, 100_000)
    if status != pic.PIC_OK:
        raise RuntimeError(pic.pic_last_error(None))
    return phi


def _exact_field(case, seed):
    """The 7-point problem solved by its own eigenvectors: Fourier in x and y, sines in z."""
    wl = _bare(case)
    nx, ny, nz = wl.nx, wl.ny, wl.nz
    rho = _density(nx, ny, nz, seed, wl.h)
    b = rho[1:nz] * (wl.h ** 2 / W.EPS0)
    b[0] += wl.phi_cathode
    b[-1] += wl.phi_anode
    k = torch.arange(1, nz, dtype=torch.float64, device="cuda")
    S = math.sqrt(2.0 / nz) * torch.sin(math.pi / nz * k[:, None] * k[None, :])

    def lam(n):
        return 2 - 2 * torch.cos(2 * math.pi * torch.arange(n, dtype=torch.float64, device="cuda") / n)

    f = torch.fft.fft2(torch.einsum("ab,byx->ayx", S, b))
    f /= (2 - 2 * torch.cos(math.pi * k / nz))[:, None, None] + lam(ny)[None, :, None] + lam(nx)[None, None, :]
    phi = torch.empty((nz + 1, ny, nx), dtype=torch.float64, device="cuda")
    phi[1:nz] = torch.einsum("ab,byx->ayx", S, torch.fft.ifft2(f).real)
    phi[0], phi[nz] = wl.phi_cathode, wl.phi_anode
    return phi


# ---------------------------------------------------------------------------
# the network of the learned warm start
# ---------------------------------------------------------------------------
def _network_inputs(case, seed):
    """He-normal weights and the two channels the network meets: a residual of unit size that is rough like
    particle noise, and the position between the electrodes (nothing on the anode plane)."""
    g = _generator(seed)
    shapes = pic.UNET_WEIGHT_SHAPES
    w = [torch.randn(s, generator=g, device="cuda", dtype=torch.float64) * math.sqrt(2.0 / (math.prod(s) / s[0])) for s in shapes]
    D, H, Wd = case["D"], case["H"], case["W"]
    r = torch.randn((D, H, Wd), generator=g, device="cuda")
    r = r + 0.5 * (r.roll(1, 1) + r.roll(1, 2))
    r[-1] = 0
    x = torch.stack([r / r.square().mean().sqrt(), (torch.arange(1, D + 1, device="cuda") / D)[:, None, None].expand(D, H, Wd)])
    dy = torch.randn((D, H, Wd), generator=g, device="cuda") / (D * H * Wd)
    return [t.to(torch.float32) for t in w], x.contiguous(), dy


def _prepare_network(case, seed):
    w, x, dy = _network_inputs(case, seed)
    net = pic.UNet(case["D"], case["H"], case["W"], weights=torch.cat([t.reshape(-1) for t in w]).cpu().numpy())
    return {"case": case, "net": net, "x": x, "dy": dy}


def _run_forward(s):
    return s["net"].forward(s["x"])


def _run_gradient(s):
    net = s["net"]
    y = net.forward(s["x"])
    return {"y": y, "grads": net.backward(s["dy"])}


def _conv(x, w):
    """3x3x3 convolution, zero padding, as the sum over its 27 taps."""
    c, D, H, Wd = x.shape
    p = torch.zeros((c, D + 2, H + 2, Wd + 2), dtype=x.dtype, device=x.device)
    p[:, 1:-1, 1:-1, 1:-1] = x
    y = torch.zeros((w.shape[0], D * H * Wd), dtype=x.dtype, device=x.device)
    for a in range(3):
        for b in range(3):
            for d in range(3):
                y.addmm_(w[:, :, a, b, d], p[:, a:a + D, b:b + H, d:d + Wd].reshape(c, -1))
    return y.reshape(-1, D, H, Wd)


def _exact_forward(case, seed):
    w, x, _ = _network_inputs(case, seed)
    w, x = [t.double() for t in w], x.double()

    def block(x, k):
        return _conv(_conv(x, w[k]).relu_(), w[k + 1]).relu_()

    def down(x):
        return torch.nn.functional.avg_pool3d(x, 2)

    def up(x):
        return x.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)

    e0 = block(x, 0)
    e1 = block(down(e0), 2)
    e2 = block(down(e1), 4)
    d = block(down(e2), 6)
    for skip, k in ((e2, 8), (e1, 10), (e0, 12)):
        d = block(torch.cat([up(d), skip]), k)
    return torch.einsum("oc,cdhw->dhw", w[14], d)


def exact(case, seed):
    if case["kind"] in ("solve", "static"):
        return _exact_field(case, seed)
    if case["kind"] == "forward":
        return _exact_forward(case, seed)
    if case["kind"] == "gradient":  # the gradients meet every ReLU that 16 bits decide otherwise: no such value
        return {"y": _exact_forward(case, seed), "grads": None}
    return None  # a run of the plasma: its draws and collisions have no closed form


# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        return _prepare_step(case, seed)
    if kind == "ensemble":
        return _prepare_ensemble(case, seed)
    if kind == "coupled":
        return _prepare_coupled(case, seed)
    if kind == "solve":
        return _prepare_solve(case, seed)
    if kind == "static":
        return _prepare_static(case, seed)
    return _prepare_network(case, seed)


def run(state):
    kind = state["case"]["kind"]
    if kind == "step":
        return _run_step(state)
    if kind == "ensemble":
        return _run_ensemble(state)
    if kind == "coupled":
        return _run_coupled(state)
    if kind == "solve":
        return state["sim"].solve(state["rho"])[0]
    if kind == "static":
        return _run_static(state)
    return _run_forward(state) if kind == "forward" else _run_gradient(state)


def _step_work(nodes, particles, steps, mixed):
    """Per step: every particle read and written once (position, velocity, identifier), the charge density and
    the potential written and read once. Per particle a push, a gather and a deposit (about 100 operations),
    per node the 7-point operator."""
    per_particle, per_node = (64, 16) if mixed else (104, 32)
    return {"bytes": steps * (particles * per_particle + nodes * per_node), "flops": steps * (100 * particles + 14 * nodes)}


def work(case):
    kind = case["kind"]
    if kind in ("step", "coupled"):
        nodes = case["nx"] * case["ny"] * (case["nz"] + 1)
        return _step_work(nodes, case["particles"], case["steps"], case.get("precision") != "fp64")
    if kind == "ensemble":
        each = [_step_work(nx * ny * (nz + 1), n, case["steps"], True) for nx, ny, nz, n in _members(case)]
        return {k: sum(e[k] for e in each) for k in ("bytes", "flops")}
    if kind in ("solve", "static"):
        nodes = case["nx"] * case["ny"] * (case["nz"] + 1)
        return {"bytes": 16 * nodes, "flops": 14 * nodes}
    voxels = case["D"] * case["H"] * case["W"]
    level = {"e0": 0, "e1": 1, "e2": 2, "e3": 3, "d2": 2, "d1": 1, "d0": 0}
    flops = sum(2 * 27 * ci * co * (voxels >> (3 * level[name[:2]])) for name, ci, co in pic.UNET_LAYERS)
    weights = 4 * sum(math.prod(s) for s in pic.UNET_WEIGHT_SHAPES)
    if kind == "forward":
        return {"bytes": 12 * voxels + weights, "flops": flops}
    return {"bytes": 16 * voxels + 2 * weights, "flops": 3 * flops}
