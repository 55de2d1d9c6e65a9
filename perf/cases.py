"""The work this framework is used for, as cases that can be timed and checked.

Every case is one pass through the public entry points of
``paper_1011_4046_gb300.sp``: an evolution call from an initial slice (split
tiling, 4-cube lattice, whole-grid sweep, the no-allocation sweep, a batch of
simulations), the diagnostics of a stored state, and the training and the
evaluation of the region cost model.  Sizes and parameters are those of the
repository's workloads (32^3 plain method, 128^3 and larger matter-era
networks, the batched simulations) or generic ones between them.
"""
import math

import numpy as np
import torch

from paper_1011_4046_gb300 import inputs, sp

MAX_UPDATES = 768 ** 3 * 65  # site-updates of the largest listed case


def listed():
    return [
        # the plain method: a small flat-space field through split regions of base 8;
        # 64 steps are 16 bands of dependent phases, so latency decides
        {"name": "plain-32", "kind": "split", "nx": 32, "ny": 32, "nz": 32, "steps": 64, "nu": 0, "base": 8, "damp": 0},
        # a caller that may not allocate advances a small field a few steps at a time
        {"name": "noalloc-48", "kind": "noalloc", "nx": 48, "ny": 40, "nz": 36, "steps": 16, "nu": 2, "damp": 0},
        # the matter-era network of ordinary size (it fits L2) through split regions of base 16 ...
        {"name": "split-128", "kind": "split", "nx": 128, "ny": 128, "nz": 128, "steps": 128, "nu": 2, "base": 16,
         "damp": 0},
        # ... and through the 4-cube lattice, a whole run of it
        {"name": "lattice-128", "kind": "lattice", "nx": 128, "ny": 128, "nz": 128, "steps": 256, "nu": 2, "base": 16,
         "damp": 0},
        # 64 uneven simulations in one call, default bases
        {"name": "batch-64", "kind": "batch", "sims": 64, "first": 0, "steps": 64},
        # the damped network: velocity discarded for half the call, then free steps
        {"name": "lattice-512", "kind": "lattice", "nx": 512, "ny": 512, "nz": 512, "steps": 64, "nu": 2, "base": 16,
         "damp": 32},
        # the large volume: state far beyond L2, an odd step count (diagnostics every 64 steps, one more step)
        {"name": "lattice-768", "kind": "lattice", "nx": 768, "ny": 768, "nz": 768, "steps": 65, "nu": 2, "base": 16,
         "damp": 0},
        # whole-grid sweep: sides that no region base divides, radiation era
        {"name": "sweep-ragged", "kind": "sweep", "nx": 150, "ny": 77, "nz": 131, "steps": 50, "nu": 1, "damp": 0},
        # whole-grid sweep of a large volume
        {"name": "sweep-512", "kind": "sweep", "nx": 512, "ny": 512, "nz": 512, "steps": 32, "nu": 2, "damp": 0},
        # energy terms and string length of a large stored state, taken every so many steps of a run
        {"name": "diag-512", "kind": "diag", "nx": 512, "ny": 512, "nz": 512, "nu": 2},
        # the cost model trained on the regions of a traced run, minibatches of 256
        {"name": "cost-train", "kind": "train", "n": 16384, "epochs": 2, "batch": 256},
        # every region of a large call ranked by the cost model
        {"name": "cost-predict", "kind": "predict", "n": 1 << 20},
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["split", "lattice", "lattice", "sweep", "sweep", "noalloc", "batch", "diag", "train", "predict"])
    if kind == "train":
        n, batch = _log(rng, 500, 32768), _log(rng, 32, 512)
        return {"kind": kind, "n": n, "batch": batch, "epochs": max(1, min(4, 192 * batch // n))}
    if kind == "predict":
        return {"kind": kind, "n": _log(rng, 1000, 1 << 21)}
    if kind == "batch":
        sims = rng.randint(3, 24)
        return {"kind": kind, "sims": sims, "first": rng.randint(0, 64 - sims), "steps": rng.randint(16, 96)}
    nu = rng.choice([0, 1, 2, 2])
    while True:
        if kind == "split":
            base = rng.choice([8, 16, 16])
            n = [base * _log(rng, 2, 240 // base) for _ in range(3)]
            steps = rng.randint(8, 160)
        elif kind == "lattice":
            base = rng.choice([8, 12, 16, 16, 16, 20])
            n = [base * _log(rng, 2, 512 // base) for _ in range(3)]
            steps = rng.randint(8, 160)
        elif kind == "noalloc":
            n = [_log(rng, 8, 96) for _ in range(3)]
            steps = _log(rng, 1, 128)
        elif kind == "sweep":
            n = [_log(rng, 16, 512) for _ in range(3)]
            steps = _log(rng, 1, 128)
        else:
            n = [_log(rng, 16, 512) for _ in range(3)]
            steps = 1
        sites = n[0] * n[1] * n[2]
        if sites * steps <= MAX_UPDATES and (kind != "noalloc" or sites <= sp.SP_NOALLOC_MAX_SITES):
            break
    case = {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "nu": nu}
    if kind != "diag":
        case.update(steps=steps, damp=rng.choice([0, 0, steps // 3]))
    if kind in ("split", "lattice"):
        case["base"] = base
    return case


# ---------------------------------------------------------------- inputs
def _physics(case):
    """The workloads' constants; tau_ref is the end of the call, where a = 1."""
    nu, steps = case["nu"], case.get("steps", 1)
    tau0 = 10.0 if nu > 0 else 1.0
    return {"dx": 1.0, "dt": 0.25, "lam": 2.0, "eta": 1.0, "nu": float(nu), "tau0": tau0, "tau_ref": tau0 + 0.25 * steps,
            "damp_steps": case.get("damp", 0)}


def _field(n, nu, gen):
    """phi (nz, ny, nx): random phases in an expanding era, Gaussian of
    standard deviation 0.3 per component in flat space."""
    shape = (n[2], n[1], n[0])
    if nu > 0:
        theta = torch.rand(shape, generator=gen, device="cuda") * (2.0 * math.pi)
        return torch.polar(torch.ones_like(theta), theta)
    return torch.view_as_complex(0.3 * torch.randn(shape + (2,), generator=gen, device="cuda"))


def _sims(case):
    """(n, nu) of every simulation of an evolution case."""
    if case["kind"] == "batch":
        return [((n, n, n), nu) for _, n, nu in inputs.batched_workload(64)[case["first"]:case["first"] + case["sims"]]]
    return [((case["nx"], case["ny"], case["nz"]), case["nu"])]


def _initial(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return [_field(n, nu, gen) for n, nu in _sims(case)]


def _stored_state(case, seed):
    """A state such as a run leaves: random phases smoothed along each axis
    (strings, gradients), velocities of the same size."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n = (case["nx"], case["ny"], case["nz"])
    phi = _field(n, case["nu"], gen)
    for axis in range(3):
        phi = 0.5 * phi + 0.5 * torch.roll(phi, 1, axis)
    pic = torch.zeros(phi.shape + (2,), dtype=torch.complex64, device="cuda")
    pic[..., 0] = 0.2 * _field(n, case["nu"], gen)
    return phi.contiguous(), pic


def _samples(case, seed):
    """Region features as the library records them (bits of the type, sizes,
    field averages) and the log of a region time that depends on them."""
    r = np.random.RandomState(seed)
    n = case["n"]
    x = r.rand(n, sp.SP_MODEL_FEATURES).astype(np.float32)
    x[:, :3] = x[:, :3] < 0.5
    x[:, 3] = x[:, :3].sum(1) / 3.0
    x[:, 4] = np.where(x[:, 4] < 0.5, 0.5, 1.0)
    y = (1.5 + 0.4 * x[:, 3] + 0.6 * x[:, 4] + 0.2 * x[:, 13] * x[:, 10] + 0.05 * r.randn(n)).astype(np.float32)
    return x, y


_LAYERS = ((64, 16), (64, 64), (1, 64))


def _weights(seed):
    r = np.random.RandomState(seed + 77)
    out = []
    for fan_out, fan_in in _LAYERS:
        out += [r.uniform(-1.0, 1.0, fan_out * fan_in) * math.sqrt(6.0 / fan_in), np.zeros(fan_out)]
    return np.concatenate(out).astype(np.float32)


# ---------------------------------------------------------------- the passes
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("train", "predict"):
        x, y = _samples(case, seed)
        m = sp.Model(seed=0)
        theta = _weights(seed)
        m.set_params(theta)
        return {"case": case, "m": m, "theta": theta, "x": torch.from_numpy(x).cuda(), "y": torch.from_numpy(y).cuda(),
                "out": torch.empty(case["n"], device="cuda")}
    if kind == "diag":
        n = (case["nx"], case["ny"], case["nz"])
        phi, pic = _stored_state(case, seed)
        g = sp.Grid([sp.make_params(n, **_physics(case))], states=[(phi, pic)])
        return {"case": case, "g": g}
    fields = _initial(case, seed)
    sims = _sims(case)
    params = [sp.make_params(n, **_physics({**case, "nu": nu})) for n, nu in sims]
    sites = [f.numel() for f in fields]
    if kind == "noalloc":
        phi, pic = fields[0].clone(), torch.zeros(fields[0].shape + (2,), dtype=torch.complex64, device="cuda")
        return {"case": case, "p": params[0], "phi0": fields[0], "phi": phi, "pic": pic}
    # one pool for the states of all simulations, and the initial slice of each
    # in the library's layout (phi, then (pi, c) = 0)
    phi = torch.empty(sum(sites), dtype=torch.complex64, device="cuda")
    pic = torch.empty(sum(sites), 2, dtype=torch.complex64, device="cuda")
    states, start, at = [], [], 0
    for f, s in zip(fields, sites):
        states.append((phi[at:at + s], pic[at:at + s]))
        at += s
        start.append(torch.zeros(3 * s, dtype=torch.complex64, device="cuda"))
        start[-1][:s] = f.reshape(-1)
    del fields
    torch.cuda.synchronize()
    g = sp.Grid(params, states=states, stream=torch.cuda.Stream())
    if kind == "split":
        g.plan(base_B=case["base"])
    elif kind == "lattice":
        g.plan(base_B=case["base"], shape=sp.SP_SHAPE_LATTICE)
    elif kind == "batch":
        g.plan()
    return {"case": case, "g": g, "start": start, "phi": phi, "pic": pic}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "train":
        m = state["m"]
        m.set_params(state["theta"])  # a new fit (the optimiser starts afresh)
        losses = m.train(state["x"].data_ptr(), state["y"].data_ptr(), case["n"], epochs=case["epochs"],
                         batch=case["batch"], lr=1e-3, order_seed=1)
        params, thresholds = m.params()
        return {"losses": losses, "params": params, "thresholds": thresholds}
    if kind == "predict":
        state["m"].predict(state["x"].data_ptr(), case["n"], state["out"].data_ptr())
        return {"y": state["out"]}
    if kind == "diag":
        return state["g"].diag(0)
    if kind == "noalloc":
        phi, pic = state["phi"], state["pic"]
        phi.copy_(state["phi0"])
        pic.zero_()
        rc = sp.sp_sweep_noalloc(state["p"], phi.data_ptr(), pic.data_ptr(), 0, case["steps"],
                                 torch.cuda.current_stream().cuda_stream)
        if rc != sp.SP_OK:
            raise sp.SpError(rc, "sp_sweep_noalloc")
    else:
        g, phi, pic = state["g"], state["phi"], state["pic"]
        for sim, buf in enumerate(state["start"]):  # the initial slice, then the whole run from level 0
            rc = sp.sp_write_surface(g.h, sim, sp.SP_SURF_STATE, buf.data_ptr(), 8 * buf.numel(), 1)
            if rc != sp.SP_OK:
                raise sp.SpError(rc, "sp_write_surface")
        g.evolve(case["steps"], sp.SP_RESTART | (sp.SP_MONOLITHIC if kind == "sweep" else 0))
    return {"phi": phi, "pi": pic[..., 0], "c": pic[..., 1]}


def work(case):
    kind = case["kind"]
    flops = 2 * (16 * 64 + 64 * 64 + 64)  # of the cost model per sample, forward
    if kind == "predict":
        return {"bytes": 68.0 * case["n"], "flops": float(flops) * case["n"]}
    if kind == "train":
        samples = case["n"] * case["epochs"]
        return {"bytes": 68.0 * samples, "flops": 3.0 * flops * samples}
    sites = float(sum(n[0] * n[1] * n[2] for n, _ in _sims(case)))
    if kind == "diag":
        return {"bytes": 24.0 * sites, "flops": 80.0 * sites}
    # the initial slice read once, the final one written once; 41 flops per site-update
    return {"bytes": 48.0 * sites, "flops": 41.0 * sites * case["steps"]}


# ---------------------------------------------------------------- 64-bit values
def _evolve64(phi, q, steps):
    phi = phi.to(torch.complex128)
    pi = torch.zeros_like(phi)
    for k in range(steps):
        damping = k < q["damp_steps"]
        tau = q["tau0"] + (0.0 if damping else (k - q["damp_steps"]) * q["dt"])
        a = (tau / q["tau_ref"]) ** q["nu"]
        d = 1.0 if damping else q["nu"] * q["dt"] / tau
        f = phi * -6.0
        for axis in range(3):
            f += torch.roll(phi, 1, axis)
            f += torch.roll(phi, -1, axis)
        f /= q["dx"] ** 2
        f -= (a * a * q["lam"] * (phi.real ** 2 + phi.imag ** 2 - q["eta"] ** 2)) * phi
        pi *= (1.0 - d) / (1.0 + d)
        pi += f * (q["dt"] / (1.0 + d))
        phi = phi + q["dt"] * pi
    return phi, pi


def _diag64(case, seed):
    q = _physics(case)
    phi, pic = _stored_state(case, seed)
    kin = pic[..., 0].to(torch.complex128).abs().square().sum()
    f = phi.to(torch.complex128)
    a = (q["tau0"] / q["tau_ref"]) ** q["nu"]
    pot = (0.5 * q["lam"] * a * a * (f.real ** 2 + f.imag ** 2 - q["eta"] ** 2) ** 2).sum()
    grad = sum((torch.roll(f, -1, ax) - f).abs().square().sum() for ax in range(3)) / q["dx"] ** 2

    def crossing(u, v):
        cr = u.real * v.imag - u.imag * v.real
        ua, va = u.imag >= 0, v.imag >= 0
        return (~ua & va & (cr >= 0)).to(torch.int8) - (ua & ~va & (cr <= 0)).to(torch.int8)

    pierced, net, total = [], [], 0
    for k in range(3):
        ax_a, ax_b = 2 - (k + 1) % 3, 2 - (k + 2) % 3  # tensor axes are (z, y, x)
        p1 = torch.roll(f, -1, ax_a)
        p2 = torch.roll(p1, -1, ax_b)
        p3 = torch.roll(f, -1, ax_b)
        w = crossing(f, p1) + crossing(p1, p2) + crossing(p2, p3) + crossing(p3, f)
        pierced.append(int((w != 0).sum()))
        net.append(int(w.long().sum()))
        total += int(w.abs().long().sum())
    kin, grad, pot = float(kin), float(grad), float(pot)
    return {"level": 0, "tau": q["tau0"], "a": a, "kinetic": kin, "gradient": grad, "potential": pot,
            "total": kin + grad + pot, "pierced": pierced, "abs_winding": total, "net_winding": net,
            "string_length": float(sum(pierced)) * q["dx"]}


def _layers64(theta):
    out, o = [], 0
    for fan_out, fan_in in _LAYERS:
        out.append((theta[o:o + fan_out * fan_in].reshape(fan_out, fan_in), theta[o + fan_out * fan_in:][:fan_out]))
        o += fan_out * fan_in + fan_out
    return out


def _predict64(theta, x):
    (w1, b1), (w2, b2), (w3, b3) = _layers64(theta)
    h1 = np.maximum(x @ w1.T + b1, 0.0)
    h2 = np.maximum(h1 @ w2.T + b2, 0.0)
    return h1, h2, (h2 @ w3.T + b3)[:, 0]


def _order(seed, epoch, n):
    """Sample order of an epoch: the stable argsort of the uniforms
    2^42 + epoch 2^32 + i of the SplitMix64 stream (Steele, Lea, Flood 2014)."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + (np.uint64((1 << 42) + (epoch << 32) + 1) + np.arange(n, dtype=np.uint64)) * np.uint64(
            0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z ^= z >> np.uint64(31)
    return np.argsort(z >> np.uint64(11), kind="stable")


def _train64(case, seed):
    x, y = (v.astype(np.float64) for v in _samples(case, seed))
    theta = _weights(seed).astype(np.float64)
    m, v, losses, t = np.zeros_like(theta), np.zeros_like(theta), [], 0
    for epoch in range(case["epochs"]):
        order = _order(1, epoch, case["n"])
        for s in range(0, case["n"], case["batch"]):
            idx = order[s:s + case["batch"]]
            xb = x[idx]
            _, (w2, _), (w3, _) = _layers64(theta)
            h1, h2, yhat = _predict64(theta, xb)
            r = yhat - y[idx]
            losses.append(float(np.mean(r * r)))
            go = (2.0 / len(idx)) * r[:, None]
            g2 = go * w3 * (h2 > 0)
            g1 = (g2 @ w2) * (h1 > 0)
            g = np.concatenate([(g1.T @ xb).ravel(), g1.sum(0), (g2.T @ h1).ravel(), g2.sum(0), (go.T @ h2).ravel(),
                                go.sum(0)])
            t += 1
            m = 0.9 * m + 0.1 * g
            v = 0.999 * v + 0.001 * g * g
            theta = theta - 1e-3 * (m / (1 - 0.9 ** t)) / (np.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
    p = np.sort(_predict64(theta, x)[2])
    thresholds = np.array([p[(case["n"] - 1) * (3 - q) // 4] for q in range(3)])
    return {"losses": np.array(losses), "params": theta, "thresholds": thresholds}


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _train64(case, seed)
    if kind == "predict":
        return {"y": _predict64(_weights(seed).astype(np.float64), _samples(case, seed)[0].astype(np.float64))[2]}
    if kind == "diag":
        return _diag64(case, seed)
    runs = [_evolve64(f, _physics({**case, "nu": nu}), case["steps"]) for f, (_, nu) in zip(_initial(case, seed), _sims(case))]
    phi, pi = (torch.cat([r[i].reshape(-1) for r in runs]) for i in range(2))
    if kind == "noalloc":
        phi, pi = phi.reshape(runs[0][0].shape), pi.reshape(runs[0][1].shape)
    return {"phi": phi, "pi": pi, "c": None}  # c is the rounding carry of 32-bit sums
