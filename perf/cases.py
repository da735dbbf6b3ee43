"""Performance cases: the work that users of this framework have it do, through
its Python entry points, from the smallest run to the largest, with the same
results in 64 bits from plain torch (exact) to say how accurate they are.

Every pass starts from a fresh state (the uniform superposition, or the box
mesh's kinetic ground state), so a case can be run again on the same context.
The potential, the schedule and the network's weights are set in prepare(), as a
user's program sets them once and keeps the context; `targets` is the exception:
the surrogate's data generation loads a new potential for each call, so there the
whole call is the pass.

psi is complex64 and carries a global phase that depends on the library's
internals, so exact() gives |psi|^2 and nothing for psi itself.
"""
import math

import numpy as np
import torch

import workloads
from paper_2303_01471_gb300 import fno, lattice, qhd, surrogate


def listed():
    return [
        # The loss curve of one small instance: observables every 10 steps, as
        # trajectories are recorded and plotted.  Latency and launches count.
        {"name": "traj_64", "kind": "trajectory", "shape": "64x64", "batch": 1, "family": "wells", "wells": 8,
         "dt": 0.01, "steps": 100, "every": 10, "split": 0, "fd2": False, "own_phi": False},
        # One 128^2 instance on its own, the single-instance benchmark configuration.
        {"name": "run_128", "kind": "solve", "shape": "128x128", "batch": 1, "family": "wells", "wells": 8,
         "dt": 0.01, "steps": 200, "split": 0, "fd2": False, "own_phi": False},
        # Training targets of the surrogate: potential, schedule, evolution and
        # |psi|^2 of a batch of 128^2 instances in one call.
        {"name": "targets_128", "kind": "targets", "n": 128, "batch": 512, "dt": 0.01, "steps": 100},
        # Ragged batch: as many 128^2 as 256^2 instances, each with its own
        # schedule scale, in one persistent launch.
        {"name": "ragged", "kind": "group", "n64": 0, "n128": 256, "n256": 256, "dt": 0.01, "steps": 50},
        # One 1024^2 instance with the Rastrigin-type f (the 2-D half of the benchmark).
        {"name": "run_1024", "kind": "solve", "shape": "1024x1024", "batch": 1, "family": "rastrigin", "wells": 8,
         "dt": 0.001, "steps": 100, "split": 0, "fd2": False, "own_phi": False},
        # One 256^3 instance with 32 wells (the 3-D half of the benchmark).
        {"name": "run_256cube", "kind": "solve", "shape": "256x256x256", "batch": 1, "family": "wells", "wells": 32,
         "dt": 0.001, "steps": 20, "split": 0, "fd2": False, "own_phi": False},
        # A batch of 512^2 instances with 16 wells on the FFT path.
        {"name": "batch_512", "kind": "solve", "shape": "512x512", "batch": 16, "family": "wells", "wells": 16,
         "dt": 0.01, "steps": 50, "split": 0, "fd2": False, "own_phi": False},
        # Small boxes of uneven axes with the finite-difference kinetic operator and
        # the first-order product formula, each instance with its own e^phi.
        {"name": "box_64x16x128", "kind": "solve", "shape": "64x16x128", "batch": 5, "family": "wells", "wells": 4,
         "dt": 0.01, "steps": 50, "split": 1, "fd2": True, "own_phi": True},
        # The tensor-core transform in its FP16 hi-lo three-product form.
        {"name": "tc_512", "kind": "tc", "n": 512, "batch": 16, "wells": 16, "products": 3, "dt": 0.01, "steps": 4},
        # Surrogate inference at the evaluation batch.
        {"name": "fno_infer", "kind": "fno", "n": 128, "batch": 512, "modes": 16, "layers": 4, "hidden": 128,
         "bf16": True, "train": False},
        # Surrogate training: the gradient of one mini-batch.
        {"name": "fno_grad", "kind": "fno", "n": 128, "batch": 64, "modes": 16, "layers": 4, "hidden": 128,
         "bf16": True, "train": True},
        # Box-constrained quadratic programs on the 9^5 mesh (Sim-QHD).
        {"name": "boxqp_5d", "kind": "box", "d": 5, "r": 8, "batch": 256, "relaxed": True, "dt": 0.01, "steps": 20},
    ]


def _log_int(rng, lo, hi):
    """A whole number in [lo, hi], spread over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


MOST_POINT_STEPS = 1 << 28  # of a drawn evolution: grid points x instances x steps


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "trajectory", "targets", "group", "tc", "fno", "box"])
    if kind in ("solve", "trajectory"):
        d = rng.choice([1, 2, 2, 2, 3, 3]) if kind == "solve" else 2
        top = {1: 10, 2: 10, 3: 8}[d]
        axes = [2 ** rng.randint(3 if d == 3 else 4, top) for _ in range(d)]
        if rng.random() < 0.5:
            axes = [axes[0]] * d
        g = math.prod(axes)
        batch = _log_int(rng, 1, max(1, min(512, (1 << 24) // g)))
        steps = _log_int(rng, 10, max(10, min(100, MOST_POINT_STEPS // (g * batch))))
        case = {"kind": kind, "shape": "x".join(map(str, axes)), "batch": batch,
                "family": rng.choice(["wells", "rastrigin"]), "wells": rng.choice([4, 8, 16]),
                "dt": rng.choice([0.01, 0.001]), "steps": steps, "split": rng.choice([0, 0, 0, 1]),
                "fd2": rng.random() < 0.25, "own_phi": rng.random() < 0.25}
        if kind == "trajectory":
            case["every"] = max(1, steps // 8)
            case["steps"] = case["every"] * 8
        return case
    if kind == "targets":
        n = rng.choice([32, 64, 128, 256])
        batch = _log_int(rng, 3, min(1024, (1 << 23) // (n * n)))
        return {"kind": kind, "n": n, "batch": batch, "dt": 0.01, "steps": _log_int(rng, 20, 60)}
    if kind == "group":
        return {"kind": kind, "n64": _log_int(rng, 1, 300), "n128": _log_int(rng, 1, 150), "n256": _log_int(rng, 1, 100),
                "dt": 0.01, "steps": _log_int(rng, 20, 60)}
    if kind == "tc":
        n = rng.choice([128, 256, 512])
        return {"kind": kind, "n": n, "batch": _log_int(rng, 1, (1 << 21) // (n * n)), "wells": 16,
                "products": rng.choice([3, 10]), "dt": 0.01, "steps": rng.randint(2, 4)}
    if kind == "fno":
        train = rng.random() < 0.5
        return {"kind": kind, "n": rng.choice([64, 128]), "batch": _log_int(rng, 3, 48 if train else 300),
                "modes": rng.choice([8, 16]), "layers": rng.choice([2, 4]), "hidden": rng.choice([64, 128]),
                "bf16": True, "train": train}
    d = rng.choice([2, 3, 4, 5])
    r = rng.randint(2, {2: 16, 3: 16, 4: 12, 5: 8}[d])
    batch = _log_int(rng, 1, min(256, (1 << 23) // (r + 1) ** d))
    return {"kind": "box", "d": d, "r": r, "batch": batch, "relaxed": rng.random() < 0.7, "dt": 0.01,
            "steps": rng.randint(8, 20)}


# ------------------------------------------------------------------- inputs
def _shape(case):
    return tuple(int(n) for n in case["shape"].split("x"))


def _potentials(seed, families, shape, wells):
    """FP64 potentials (B, *shape) on the GPU and each instance's schedule scale."""
    spec = [(families[i % len(families)], 1000 * seed + i) for i in range(len(families))]
    f, sigma = workloads.batch_fast_on_device(spec, shape, "cuda", K=wells, chunk=max(1, (1 << 25) // math.prod(shape)))
    return f, sigma


def _schedules(case, sigma):
    """(c_phi, c_chi) of each instance: e^phi = c_phi / (1e-3 + t^3), e^chi = c_chi t^3."""
    return [(2.0 + (0.1 * (i % 7) if case.get("own_phi") else 0.0), 2.0 * s) for i, s in enumerate(sigma)]


def _loaded(shape, f, coefs):
    sim = qhd.QHD(shape, batch=f.shape[0])
    sim.set_potential(f)
    sim.set_schedule([qhd.Schedule(c_phi=p, c_chi=c) for p, c in coefs])
    return sim


def _boxes(case, seed):
    qb = [workloads.box_qp(1000 * seed + i, case["d"]) for i in range(case["batch"])]
    rng = np.random.default_rng(seed)
    return np.stack([q for q, _ in qb]), np.stack([b for _, b in qb]), rng.uniform(0.5, 2.0, case["batch"])


def _weights(case, seed):
    """The network's parameter blocks in the order of the library's parameter vector."""
    rng = np.random.default_rng(seed)
    c, m, h = 32, case["modes"], case["hidden"]
    blocks = [("lift_w", (c, 4), 0.5, 0), ("lift_b", (c,), 0.1, 0)]
    for l in range(case["layers"]):
        blocks += [("R%d" % l, (2 * m, m, c, c, 2), 1.0 / c ** 2, 1), ("W%d" % l, (c, c), c ** -0.5, 0),
                   ("b%d" % l, (c,), 0.1, 0)]
    blocks += [("p1_w", (h, c), c ** -0.5, 0), ("p1_b", (h,), 0.1, 0), ("p2_w", (h,), h ** -0.5, 0), ("p2_b", (1,), 0.1, 0)]
    return [(k, rng.uniform(0.0 if positive else -a, a, s).astype(np.float32)) for k, s, a, positive in blocks]


def _flat(blocks):
    """One vector, every block starting at an even offset."""
    parts = []
    for b in blocks:
        parts.append(b.reshape(-1))
        if parts[-1].numel() % 2:
            parts.append(torch.zeros(1, dtype=b.dtype, device=b.device))
    return torch.cat(parts)


def _fno_inputs(case, seed):
    fam = ["wells", "rastrigin"] * case["batch"]
    f, sigma = _potentials(seed, fam[: case["batch"]], (case["n"], case["n"]), 8)
    sigma = torch.tensor(sigma, dtype=torch.float32, device="cuda")
    # a distribution that sits in f's lowest regions, as the solver's |psi(T)|^2 does
    low = (f - f.amin((1, 2), keepdim=True)) / (f.amax((1, 2), keepdim=True) - f.amin((1, 2), keepdim=True))
    p_true = torch.softmax((-30.0 * low).flatten(1), 1).reshape(f.shape).float()
    return f, sigma, p_true


# ------------------------------------------------------------------ prepare
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("solve", "trajectory", "tc"):
        shape = (case["n"], case["n"]) if kind == "tc" else _shape(case)
        f, sigma = _potentials(seed, [case.get("family", "wells")] * case["batch"], shape, case["wells"])
        if case["batch"] == 1:
            sigma = [1.0]
        sim = _loaded(shape, f, _schedules(case, sigma))
        if kind == "tc":
            sim.set_transform(qhd.TRANSFORM_TC_DFT, case["products"])
        else:
            sim.set_splitting(qhd.SPLIT_LIE_TROTTER if case["split"] else qhd.SPLIT_STRANG)
            sim.set_kinetic(qhd.KINETIC_FD2 if case["fd2"] else qhd.KINETIC_SPECTRAL)
        return {"case": case, "sim": sim}
    if kind == "targets":
        fam = ["wells", "rastrigin"] * case["batch"]
        f, sigma = _potentials(seed, fam[: case["batch"]], (case["n"], case["n"]), 8)
        return {"case": case, "f": f, "sigma": sigma}
    if kind == "group":
        sims = []
        for k, n in enumerate((64, 128, 256)):
            if case["n%d" % n]:
                fam = (["wells", "rastrigin"] * case["n%d" % n])[: case["n%d" % n]]
                f, sigma = _potentials(3 * seed + k, fam, (n, n), 8)
                sims.append(_loaded((n, n), f, _schedules(case, sigma)))
        return {"case": case, "sims": sims, "group": qhd.Group(sims)}
    if kind == "fno":
        cfg = fno.FNOConfig(n=case["n"], width=32, modes=case["modes"], layers=case["layers"], hidden=case["hidden"],
                            act_bf16=case["bf16"])
        params = _flat([torch.from_numpy(w) for _, w in _weights(case, seed)])
        net = fno.FNO(cfg, case["batch"], train=case["train"], params=params)
        f, sigma, p_true = _fno_inputs(case, seed)
        return {"case": case, "net": net, "f": f, "sigma": sigma, "p_true": p_true}
    q, b, sigma = _boxes(case, seed)
    lat = lattice.Lattice(case["d"], case["r"], lattice.RELAXED if case["relaxed"] else lattice.CHAIN, batch=case["batch"])
    lat.set_qp(q, b)
    lat.set_schedule([qhd.Schedule(c_chi=2.0 * s) for s in sigma])
    return {"case": case, "lat": lat}


# ---------------------------------------------------------------------- run
def _distribution(psi):
    return torch.view_as_real(psi).square().sum(-1)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("solve", "tc"):
        sim = state["sim"]
        sim.reset_state()
        sim.evolve(case["steps"] * case["dt"], case["dt"])
        return {"psi": sim.psi, "p": _distribution(sim.psi)}
    if kind == "trajectory":
        sim = state["sim"]
        sim.reset_state()
        traj = sim.evolve_trajectory(case["steps"] * case["dt"], case["dt"], case["every"])
        # sums over a complex64 state: single precision is what they hold
        return {"psi": sim.psi, "p": _distribution(sim.psi), "trajectory": traj.float()}
    if kind == "targets":
        return {"p": surrogate.solver_distributions(state["f"], state["sigma"], T=case["steps"] * case["dt"], dt=case["dt"])}
    if kind == "group":
        for sim in state["sims"]:
            sim.reset_state()
        state["group"].evolve(case["steps"] * case["dt"], case["dt"])
        return {"psi": [sim.psi for sim in state["sims"]], "p": [_distribution(sim.psi) for sim in state["sims"]]}
    if kind == "fno":
        net = state["net"]
        if not case["train"]:
            return {"p": net.forward(state["f"], state["sigma"])}
        net.loss_grad(state["f"], state["sigma"], state["p_true"], want_loss=False)
        return {"grad": net.grad}
    lat = state["lat"]
    lat.reset_state(lattice.INIT_GROUND)
    lat.evolve(case["steps"] * case["dt"], case["dt"])
    psi = lat.state()
    return {"psi": psi, "p": _distribution(psi)}


# --------------------------------------------------------------------- work
def work(case):
    """Bytes: the potential (or network input and weights) in, the state and the
    distribution out.  Operations: split radix-2 transforms (5 N log2 N) and one
    complex product per phase and step; the dense products where the path is one
    by definition (tensor-core transform, box mesh, network)."""
    kind = case["kind"]

    def evolution(g, batch, steps, out):
        return {"bytes": g * batch * (8 + out), "flops": g * batch * steps * (10 * math.log2(g) + 12)}

    if kind in ("solve", "trajectory"):
        return evolution(math.prod(_shape(case)), case["batch"], case["steps"], 12)
    if kind == "targets":
        return evolution(case["n"] ** 2, case["batch"], case["steps"], 4)
    if kind == "group":
        parts = [evolution(n * n, case["n%d" % n], case["steps"], 12) for n in (64, 128, 256)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if kind == "tc":
        g = case["n"] ** 2 * case["batch"]
        return {"bytes": g * 20, "flops": g * case["steps"] * 4 * case["products"] * 8 * case["n"]}
    if kind == "fno":
        n, b, c, m, h = case["n"], case["batch"], 32, case["modes"], case["hidden"]
        layer = n * n * (2 * c * c + 2 * 4 * m * c) + n * m * 2 * (8 * 2 * m * c) + 2 * m * m * 8 * c * c
        flops = n * n * (2 * h * c + 2 * h + 8 * c) + case["layers"] * layer
        weights = 4 * case["layers"] * (4 * m * m * c * c + c * c)
        return {"bytes": b * n * n * 12 + weights * (2 if case["train"] else 1), "flops": b * flops * (3 if case["train"] else 1)}
    n, g = case["r"] + 1, (case["r"] + 1) ** case["d"]
    low = n // 2  # both kinetic operators split into a symmetric and an antisymmetric block
    line = 8 * ((n - low) ** 2 + low ** 2) / n
    return {"bytes": g * case["batch"] * 20, "flops": g * case["batch"] * case["steps"] * (case["d"] * line + 6)}


# -------------------------------------------------------------------- exact
def _coefficients(coefs, t):
    p, c = (torch.tensor(v, dtype=torch.float64, device="cuda") for v in zip(*coefs))
    return p / (1e-3 + t ** 3), c * t ** 3


def _rotation(angle):
    return torch.polar(torch.ones_like(angle), -angle)


def _evolved(case, f, coefs, every=0):
    """|psi|^2 of the split-step evolution in complex128, and every `every` steps the observables."""
    shape, batch = tuple(f.shape[1:]), f.shape[0]
    d, dt, first_order = len(shape), case["dt"], bool(case.get("split"))
    kin = torch.zeros(shape, dtype=torch.float64, device="cuda")
    for a, n in enumerate(shape):
        m = torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device="cuda")
        e = (4.0 * n * n) * torch.sin(math.pi * m / n) ** 2 if case.get("fd2") else (2.0 * math.pi * m) ** 2
        kin = kin + 0.5 * e.reshape([-1 if i == a else 1 for i in range(d)])
    col = (batch,) + (1,) * d
    axes = tuple(range(1, d + 1))
    psi = torch.full(f.shape, math.prod(shape) ** -0.5, dtype=torch.complex128, device="cuda")
    rows = []
    for j in range(case["steps"]):
        a, b = _coefficients(coefs, (j if first_order else j + 0.5) * dt)
        half = _rotation((dt if first_order else 0.5 * dt) * b.reshape(col) * f)
        psi = torch.fft.ifftn(torch.fft.fftn(psi * half, dim=axes) * _rotation(dt * a.reshape(col) * kin), dim=axes)
        if not first_order:
            psi = psi * half
        if every and (j + 1) % every == 0:
            p = torch.view_as_real(psi).square().sum(-1)
            at = np.unravel_index(f.flatten(1).argmin(1).cpu().numpy(), shape)
            r2 = torch.zeros_like(f)
            for k, n in enumerate(shape):
                x = torch.arange(n, dtype=torch.float64, device="cuda") / n
                here = torch.tensor(at[k] / n, dtype=torch.float64, device="cuda").reshape(col)
                r2 = r2 + (x.reshape([1] + [-1 if i == k else 1 for i in range(d)]) - here) ** 2
            near = (r2.sqrt() < 0.1).double()
            rows.append(torch.stack([(p * w).flatten(1).sum(1) for w in (torch.ones_like(p), f, near)], 1))
    return torch.view_as_real(psi).square().sum(-1), torch.stack(rows) if rows else None


def _box_evolved(case, seed):
    q, b, sigma = _boxes(case, seed)
    n, d, r, batch, dt = case["r"] + 1, case["d"], case["r"], case["batch"], case["dt"]
    j = np.arange(n - 1)
    link = np.sqrt((j + 1.0) * (r - j) / r) if case["relaxed"] else np.ones(n - 1)
    lam, vec = np.linalg.eigh(np.diag(link, 1) + np.diag(link, -1))
    ground = torch.tensor(np.abs(vec[:, -1]), device="cuda").to(torch.complex128)
    lam, vec = torch.tensor(lam, device="cuda"), torch.tensor(vec, device="cuda").to(torch.complex128)
    x = torch.arange(n, dtype=torch.float64, device="cuda") / r
    grid = torch.stack(torch.meshgrid(*[x] * d, indexing="ij"), -1).reshape(-1, d)
    qt, bt = torch.tensor(q, device="cuda"), torch.tensor(b, device="cuda")
    f = 0.5 * torch.einsum("gi,bij,gj->bg", grid, qt, grid) + bt @ grid.T
    psi = ground
    for _ in range(d - 1):
        psi = torch.kron(psi, ground)
    psi = psi.expand(batch, -1)
    c = torch.tensor(sigma, device="cuda") * 2.0
    for k in range(case["steps"]):
        t = (k + 0.5) * dt
        half = _rotation(0.5 * dt * t ** 3 * c[:, None] * f)
        u = (vec * torch.polar(torch.ones_like(lam), dt * 2.0 / (1e-3 + t ** 3) * (0.5 * r * r) * lam)) @ vec.T
        psi = (psi * half).reshape((batch,) + (n,) * d)
        for a in range(1, d + 1):
            psi = torch.tensordot(psi, u, dims=([a], [1])).movedim(-1, a)
        psi = psi.reshape(batch, -1) * half
    return torch.view_as_real(psi).square().sum(-1).reshape((batch,) + (n,) * d)


def _network(case, w, f, sigma):
    """log p of the Fourier neural operator in 64 bits, from its definition."""
    n, m, b = case["n"], case["modes"], f.shape[0]
    mean = f.mean((1, 2), keepdim=True)
    std = ((f * f).mean((1, 2), keepdim=True) - mean * mean).sqrt()
    x = torch.arange(n, dtype=torch.float64, device="cuda") / n
    feats = torch.stack([(f - mean) / std, sigma.double().reshape(b, 1, 1).expand_as(f),
                         x.reshape(1, n, 1).expand_as(f), x.reshape(1, 1, n).expand_as(f)], -1)
    v = feats @ w["lift_w"].T + w["lift_b"]
    kx = torch.cat([torch.arange(m), torch.arange(n - m, n)]).double().cuda()
    ex = torch.polar(torch.ones(2 * m, n, dtype=torch.float64, device="cuda"), -2.0 * math.pi * kx[:, None] * x[None])
    ky = torch.arange(m, dtype=torch.float64, device="cuda")
    ey = torch.polar(torch.ones(m, n, dtype=torch.float64, device="cuda"), -2.0 * math.pi * ky[:, None] * x[None])
    twice = torch.where(ky == 0, 1.0, 2.0).to(torch.complex128)
    for l in range(case["layers"]):
        s = torch.einsum("lx,bxkc->blkc", ex, torch.einsum("ky,bxyc->bxkc", ey, v.to(torch.complex128)))
        s = torch.einsum("blki,lkio->blko", s, torch.view_as_complex(w["R%d" % l])) * twice.reshape(1, 1, m, 1)
        s = torch.einsum("ky,bxkc->bxyc", ey.conj(), torch.einsum("lx,blkc->bxkc", ex.conj(), s)).real / (n * n)
        v = s + v @ w["W%d" % l].T + w["b%d" % l]
        if l + 1 < case["layers"]:
            v = torch.nn.functional.gelu(v)
    z = torch.nn.functional.gelu(v @ w["p1_w"].T + w["p1_b"]) @ w["p2_w"] + w["p2_b"]
    return torch.log_softmax(z.flatten(1), 1).reshape(f.shape)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "trajectory", "tc"):
        shape = (case["n"], case["n"]) if kind == "tc" else _shape(case)
        f, sigma = _potentials(seed, [case.get("family", "wells")] * case["batch"], shape, case["wells"])
        p, rows = _evolved(case, f, _schedules(case, [1.0] if case["batch"] == 1 else sigma), case.get("every", 0))
        out = {"psi": None, "p": p}
        return {**out, "trajectory": rows} if kind == "trajectory" else out
    if kind == "targets":
        fam = ["wells", "rastrigin"] * case["batch"]
        f, sigma = _potentials(seed, fam[: case["batch"]], (case["n"], case["n"]), 8)
        return {"p": _evolved(case, f, _schedules(case, sigma))[0]}
    if kind == "group":
        ps = []
        for k, n in enumerate((64, 128, 256)):
            if case["n%d" % n]:
                fam = (["wells", "rastrigin"] * case["n%d" % n])[: case["n%d" % n]]
                f, sigma = _potentials(3 * seed + k, fam, (n, n), 8)
                ps.append(_evolved(case, f, _schedules(case, sigma))[0])
        return {"psi": [None] * len(ps), "p": ps}
    if kind == "fno":
        f, sigma, p_true = _fno_inputs(case, seed)
        w = {k: torch.tensor(v, device="cuda").double().requires_grad_(case["train"]) for k, v in _weights(case, seed)}
        ps, step = [], 16  # instances at a time: the activations are large in 64 bits
        for i in range(0, case["batch"], step):
            with torch.set_grad_enabled(case["train"]):
                logp = _network(case, w, f[i:i + step], sigma[i:i + step])
                if case["train"]:
                    (-(p_true[i:i + step].double() * logp).sum() / case["batch"]).backward()
                else:
                    ps.append(logp.exp())
        return {"grad": _flat([v.grad for v in w.values()])} if case["train"] else {"p": torch.cat(ps)}
    return {"psi": None, "p": _box_evolved(case, seed)}
