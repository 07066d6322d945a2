"""What this framework is measured on: calls of its public entry points, over the range of sizes, media and options
that its users run, from one fallback step group on a small lattice to the 8192^2 workload.

A case is a dict of plain values; `kind` says which entry points it goes through:
  step     qla.Simulation.step: the time advance (Eq. 28 or Eq. 23) from a given state
  diag     qla.Simulation.diagnostics and divD: what a run records between its step calls
  batch    qla.Batch.run over lattices of uneven sizes, and the read-back of their fields
  forward  surrogate.Surrogate.forward: one call of the trained network
  train    surrogate.Surrogate.loss_grad and adam_step: one training step
Inputs (index fields, states, training pairs) come from the seed alone, on the GPU; `exact` evaluates the same call with
plain torch operations in 64 bits.
"""
import math
import os

import numpy as np
import torch

from paper_2301_13601_gb300 import qla, surrogate, surrogate_train

CHECKPOINT = os.path.join(os.path.dirname(os.path.abspath(surrogate_train.__file__)), "checkpoints",
                          "surrogate_k16.npz")


def _step(name, Nx, Ny, steps, precision="fp32", sequence="interleaved", potential="paper", families="both",
          delta=0.05):
    return {"name": name, "kind": "step", "Nx": Nx, "Ny": Ny, "steps": steps, "precision": precision,
            "sequence": sequence, "potential": potential, "families": families, "delta": delta}


def listed():
    return [
        # one fallback group of a surrogate rollout (16 steps) on the smallest lattice of the batch workload: the
        # call is a few launches long
        _step("step_256", 256, 256, 16),
        # the FP64 correctness mode on its own lattice size (the 256^2 cylinder)
        _step("fp64_256", 256, 256, 20, precision="fp64", delta=0.1),
        # odd sizes (rows that are not a multiple of 16 bytes) and an odd number of steps
        _step("step_ragged_1001x667", 1001, 667, 25, delta=0.1),
        # 16 plain steps on the surrogate's lattice: what one call of the network stands for
        _step("step_1024", 1024, 1024, 16),
        # the ellipse workload's lattice, one recording interval
        _step("step_2048", 2048, 2048, 100),
        # the paper's other operator variants (Eq. 23 order, unitary potentials) on a lattice that is not square
        _step("step_plain_unitary_1536x1000", 1536, 1000, 48, sequence="plain", potential="unitary", delta=0.3),
        # a scattering study with one polarisation: only the E_z family is stored and advanced
        _step("step_tm_4096", 4096, 4096, 40, families="TM", delta=0.1),
        # the large workload's lattice (three cylinders at 8192^2)
        _step("step_8192", 8192, 8192, 20, delta=0.02),
        # the records between two step calls: energy, div B and div D of a large state
        {"name": "diag_4096", "kind": "diag", "Nx": 4096, "Ny": 4096},
        # a parameter study: ten independent lattices of the batch workload's sizes, fields read back at the end
        {"name": "batch_10", "kind": "batch", "count": 10, "side_min": 256, "side_max": 1024, "steps": 400},
        # one call of the trained network on the lattice it is evaluated on
        {"name": "forward_1024", "kind": "forward", "H": 1024, "W": 1024, "nimg": 1},
        # one training step at the training script's lattice and batch size
        {"name": "train_512x256x4", "kind": "train", "H": 256, "W": 512, "nimg": 4},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 7 + ["fp64", "diag", "batch", "forward", "train"])
    if kind in ("step", "fp64"):
        f64 = kind == "fp64"
        Nx, Ny = _log(rng, 64, 512 if f64 else 6144), _log(rng, 48, 512 if f64 else 6144)
        if rng.random() < 0.6:
            Nx = max(64, Nx // 8 * 8)  # most lattices are a multiple of 8 wide
        steps = max(2, min(_log(rng, 8, 120), int(6e8 / (Nx * Ny))))
        return {"kind": "step", "Nx": Nx, "Ny": Ny, "steps": steps, "precision": "fp64" if f64 else "fp32",
                "sequence": rng.choice(["interleaved", "interleaved", "plain"]),
                "potential": rng.choice(["paper", "paper", "unitary"]),
                "families": rng.choice(["both", "both", "TM", "TE"]), "delta": rng.choice([0.02, 0.05, 0.1, 0.3])}
    if kind == "diag":
        return {"kind": "diag", "Nx": _log(rng, 200, 6144), "Ny": _log(rng, 200, 6144)}
    if kind == "batch":
        lo = rng.choice([256, 384])
        return {"kind": "batch", "count": rng.randint(3, 10), "side_min": lo, "side_max": rng.choice([512, 768, 1024]),
                "steps": 4 * rng.randint(50, 100)}
    H, W = _log(rng, 64, 1024), 128 * rng.randint(1, 8)
    return {"kind": kind, "H": H, "W": W, "nimg": rng.randint(1, 2 if kind == "train" else 3)}


# ---- inputs -----------------------------------------------------------------
DEV = "cuda"


def _grid(Nx, Ny):
    y = torch.arange(Ny, dtype=torch.float64, device=DEV)[:, None]
    x = torch.arange(Nx, dtype=torch.float64, device=DEV)[None, :]
    return x, y


def _medium(Nx, Ny, r):
    """Index fields (3, Ny, Nx) of one to three tanh-edged ellipses in vacuum."""
    x, y = _grid(Nx, Ny)
    side = min(Nx, Ny)
    n = torch.ones(3, Ny, Nx, dtype=torch.float64, device=DEV)
    for _ in range(int(r.integers(1, 4))):
        a, b = r.uniform(0.05, 0.25, 2) * side
        cx, cy = r.uniform(0.45, 0.75) * Nx, r.uniform(0.3, 0.7) * Ny
        ang, w = r.uniform(0.0, math.pi), max(2.0, side / 256.0)
        dx, dy = x - cx, y - cy
        u, v = math.cos(ang) * dx + math.sin(ang) * dy, -math.sin(ang) * dx + math.cos(ang) * dy
        d = (torch.sqrt((u / a) ** 2 + (v / b) ** 2) - 1.0) * math.sqrt(a * b)
        prof = 0.5 * (1.0 - torch.tanh(d / w))
        del dx, dy, u, v, d
        for i in range(3):
            n[i] = torch.maximum(n[i], 1.0 + (r.uniform(1.0, 3.0) - 1.0) * prof)
    return n


def _pulses(Nx, Ny, r, families="both", dtype=torch.float32, shift=0.0):
    """State (6, Ny, Nx): a pulse of each advanced polarisation, its amplitude slowly varying along y."""
    x, y = _grid(Nx, Ny)
    q = torch.zeros(6, Ny, Nx, dtype=dtype, device=DEV)
    for fam, (e, b, sgn) in (("TM", (2, 4, -1.0)), ("TE", (1, 5, 1.0))):
        x0, sig, amp = r.uniform(0.2, 0.8) * Nx, r.uniform(0.02, 0.06) * Nx, r.uniform(0.5, 1.5)
        k, ph = int(r.integers(1, 4)), r.uniform(0.0, 2 * math.pi)
        if families not in ("both", fam):
            continue
        d = x - (x0 + shift)
        d = d - Nx * torch.floor(d / Nx + 0.5)
        g = amp * torch.exp(-d * d / (2.0 * sig * sig)) * (1.0 + 0.2 * torch.cos(2 * math.pi * k * y / Ny + ph))
        q[e] = g.to(dtype)
        q[b] = (sgn * g).to(dtype)
    return q


def _step_inputs(c, seed):
    r = np.random.default_rng([seed, 1])
    n = _medium(c["Nx"], c["Ny"], r)
    q = _pulses(c["Nx"], c["Ny"], r, c.get("families", "both"),
                torch.float64 if c.get("precision") == "fp64" else torch.float32)
    if c["kind"] == "diag":  # a state with every component and a divergence, as a run in a medium has
        x, y = _grid(c["Nx"], c["Ny"])
        for k in range(6):
            a = r.uniform(0.05, 0.3)
            kx, ky, ph = int(r.integers(1, 9)), int(r.integers(1, 9)), r.uniform(0.0, 6.0)
            q[k] += (a * torch.cos(2 * math.pi * (kx * x / c["Nx"] + ky * y / c["Ny"]) + ph)).to(q.dtype)
    return n, q


def _batch_sides(c, k):
    side = c["side_min"] + (c["side_max"] - c["side_min"]) * k // max(1, c["count"] - 1)
    return side // 4 * 4, side - side * (k % 4) // 12  # Ny down to three quarters of the width


def _batch_inputs(c, seed):
    r = np.random.default_rng([seed, 2])
    out = []
    for k in range(c["count"]):
        Nx, Ny = _batch_sides(c, k)
        n = _medium(Nx, Ny, r)
        steps = c["steps"] // 4 * 4 - 4 * (k % 3)
        out.append((n, steps, ("Ez", "Ey")[k % 2], 0.125 * Nx, r.uniform(0.02, 0.05) * Nx))
    return out


def _net_inputs(c, seed):
    """q_in, q_target (nimg, 6, H, W) and n (nimg, 3, H, W): pulses, and the same moved on by the 0.8 cells that 16
    steps of delta 0.05 advance a wave in vacuum."""
    r = np.random.default_rng([seed, 3])
    q, n, t = [], [], []
    for _ in range(c["nimg"]):
        n.append(_medium(c["W"], c["H"], r).float())
        s = int(r.integers(1 << 30))
        q.append(_pulses(c["W"], c["H"], np.random.default_rng(s)))
        t.append(_pulses(c["W"], c["H"], np.random.default_rng(s), shift=0.8))
    return torch.stack(q), torch.stack(n), torch.stack(t)


def _params():
    return surrogate_train.load_checkpoint(CHECKPOINT)[0]


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "step":
        n, q = _step_inputs(c, seed)
        sim = qla.Simulation(*n.cpu().numpy(), c["delta"], precision=c["precision"], sequence=c["sequence"],
                             potential=c["potential"], families=c["families"])
        sim.set_fields(q.cpu().numpy())
        return {"kind": kind, "sim": sim, "steps": c["steps"]}
    if kind == "diag":
        n, q = _step_inputs(c, seed)
        sim = qla.Simulation(*n.cpu().numpy(), 0.05)
        sim.set_fields(q.cpu().numpy())
        return {"kind": kind, "sim": sim}
    if kind == "batch":
        inst = [{"n": n.cpu().numpy(), "delta": 0.05, "nsteps": steps, "pulse": (pol, x0, sigma, 1.0)}
                for n, steps, pol, x0, sigma in _batch_inputs(c, seed)]
        return {"kind": kind, "batch": qla.Batch(inst), "count": c["count"]}
    q, n, t = _net_inputs(c, seed)
    net = surrogate.Surrogate(c["H"], c["W"], nimg=c["nimg"], train=kind == "train")
    net.set_params(_params())
    return {"kind": kind, "net": net, "q": q, "n": n, "t": t, "out": torch.empty_like(q)}


def run(state):
    kind = state["kind"]
    if kind == "step":
        sim = state["sim"]
        sim.step(state["steps"])
        torch.cuda.current_stream().wait_stream(sim.stream)  # the caller reads the state on its own stream
        return sim.state_tensor()
    if kind == "diag":
        d = state["sim"].diagnostics()
        div, dmax, big = state["sim"].divD()
        return [d["energy"], d["div_l2_sq"], d["div_max"], d["b_max"], div, dmax, big, int(d["nonfinite"])]
    if kind == "batch":
        state["batch"].run()
        return [state["batch"].get_fields(i) for i in range(state["count"])]
    if kind == "forward":
        state["net"].forward(state["q"], state["n"], state["out"])
        return state["out"]
    loss, grad = state["net"].loss_grad(state["q"], state["n"], state["t"], want_loss=True, want_grad=True)
    state["net"].adam_step(1e-5)
    return [loss, grad]


# ---- the work a pass cannot do without ----------------------------------------
def _step_flops(c_sites, steps, families, unitary):
    # per family and step: 16 collisions and 4 potential applications; a collision is a plane rotation (4 products, 2
    # sums), a printed potential row 2 products and 1 sum, a unitary one a rotation
    fam = 2 if families == "both" else 1
    return c_sites * steps * fam * (16 * 6 + 4 * (6 if unitary else 3))


def work(case):
    c, kind = case, case["kind"]
    if kind == "step":
        P, es = c["Nx"] * c["Ny"], 8 if c["precision"] == "fp64" else 4
        comps, idx = {"both": (6, 3), "TM": (3, 1), "TE": (3, 2)}[c["families"]]
        return {"bytes": P * es * (2 * comps + idx),  # state in, state out, index fields
                "flops": _step_flops(P, c["steps"], c["families"], c["potential"] == "unitary")}
    if kind == "diag":  # diagnostics read 6 planes; div D 3 planes and 3 index fields (32 bits each)
        P = c["Nx"] * c["Ny"]
        return {"bytes": P * 4 * 12, "flops": P * (12 + 7 + 6 + 9 + 6)}
    if kind == "batch":
        b = f = 0
        for k in range(c["count"]):
            Nx, Ny = _batch_sides(c, k)
            P = Nx * Ny
            b += P * 4 * 15
            f += _step_flops(P, c["steps"] // 4 * 4 - 4 * (k % 3), "both", False)
        return {"bytes": b, "flops": f}
    NP = c["H"] * c["W"] * c["nimg"]
    macs = 9 * sum(i * o for i, o in surrogate.LAYERS)
    wb = 4 * surrogate.param_count()
    if kind == "forward":  # q, n in, q out
        return {"bytes": NP * 4 * 15 + wb, "flops": 2 * macs * NP}
    # forward, weight gradient and input gradient (none for the first layer); the six layers' activations written
    # forward and read backward in 16 bits
    back = 2 * macs - 9 * surrogate.LAYERS[0][0] * surrogate.LAYERS[0][1]
    return {"bytes": NP * (4 * 15 + 2 * 2 * 5 * 64) + 8 * wb, "flops": 2 * (macs + back) * NP}


# ---- the same calls in 64 bits -------------------------------------------------
_FAMILIES = {  # hub, x-partner, y-partner; theta of C_X, C_Y; beta of V_X, V_Y; orientations of C_X, C_Y, V_X, V_Y;
    # whether the potential rows write the hub
    "TM": (2, 4, 3, 2, 2, 2, 3, -1, +1, -1, +1, False),
    "TE": (5, 1, 0, 1, 0, 0, 1, +1, -1, +1, -1, True),
}


def _direction(h, p, cs, sn, sg, dim, pot):
    """The sixteen operators of one direction (Eq. 18, Eq. 20), `pot` after the eighth and the last."""
    def c(h, p, dag):
        s = -sg if dag else sg
        return torch.addcmul(cs * h, sn, p, value=s), torch.addcmul(cs * p, sn, h, value=-s)

    def up(a):  # q(r) <- q(r + 1)
        return torch.roll(a, -1, dim)

    def down(a):
        return torch.roll(a, 1, dim)

    h, p = c(h, p, True)
    p = down(p)
    h, p = c(h, p, False)
    p = up(p)
    h, p = c(h, p, True)
    h = up(h)
    h, p = c(h, p, False)
    h = down(h)
    h, p = pot(h, p)
    h, p = c(h, p, False)
    p = up(p)
    h, p = c(h, p, True)
    p = down(p)
    h, p = c(h, p, False)
    h = down(h)
    h, p = c(h, p, True)
    h = up(h)
    return pot(h, p)


def _advance(n, q, delta, steps, interleaved, unitary, families):
    """`steps` time steps of q (6, Ny, Nx) in the medium n, every operator a sweep over the lattice."""
    nx, ny, nz = n
    theta = [delta / (4.0 * v) for v in n]

    def beta(v, dim):
        return delta * delta * (torch.roll(v, -1, dim) - torch.roll(v, 1, dim)) / (2.0 * delta) / (v * v)

    X, Y = 1, 0
    scale = (0.5 if interleaved else 1.0) * (0.5 if unitary else 1.0)
    pairs = lambda a: (torch.cos(a), torch.sin(a))  # noqa: E731
    th = [pairs(t) for t in theta]
    be = [pairs(scale * b) for b in (beta(ny, X), beta(nx, Y), beta(nz, X), beta(nz, Y))]
    q = [v.double().clone() for v in q]
    for fam, (H, PX, PY, tx, ty, bx, by, sgx, sgy, sx, sy, hub) in _FAMILIES.items():
        if families not in ("both", fam):
            continue
        h, px, py = q[H], q[PX], q[PY]

        def v(h, p, b, sg):
            cb, sb = be[b]
            if hub:
                return torch.addcmul(cb * h, sb, p, value=sg), (torch.addcmul(cb * p, sb, h, value=-sg) if unitary
                                                                else p)
            return (torch.addcmul(cb * h, sb, p, value=-sg) if unitary else h), torch.addcmul(cb * p, sb, h, value=sg)

        inside = (lambda b, sg: lambda h, p: v(h, p, b, sg)) if interleaved else (lambda b, sg: lambda h, p: (h, p))
        for _ in range(steps):
            h, px = _direction(h, px, *th[tx], sgx, X, inside(bx, sx))
            h, py = _direction(h, py, *th[ty], sgy, Y, inside(by, sy))
            if not interleaved:
                h, px = v(h, px, bx, sx)
                h, py = v(h, py, by, sy)
        q[H], q[PX], q[PY] = h, px, py
    return torch.stack(q)


def _gelu(x):
    return 0.5 * x * (1.0 + torch.tanh(math.sqrt(2.0 / math.pi) * (x + 0.044715 * x ** 3)))


def _network(x, n, params):
    import torch.nn.functional as F

    def conv(a, k):
        w, b = params[k]
        pad = F.pad(a, (1, 1, 1, 1), mode="circular")
        return sum(torch.einsum("nc,ichw->inhw", w[:, :, i, j], pad[:, :, i:i + a.shape[2], j:j + a.shape[3]])
                   for i in range(3) for j in range(3)) + b[None, :, None, None]

    a = _gelu(conv(torch.cat([x, n], 1), 0))
    for k in range(1, 5):
        a = a + _gelu(conv(a, k))
    return conv(a, 5)


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "step":
        n, q = _step_inputs(c, seed)
        return _advance(n, q, c["delta"], c["steps"], c["sequence"] == "interleaved", c["potential"] == "unitary",
                        c["families"])
    if kind == "diag":
        n, q = _step_inputs(c, seed)
        q = q.double()

        def div(u, v):
            return 0.5 * (torch.roll(u, -1, 1) - torch.roll(u, 1, 1)) + 0.5 * (torch.roll(v, -1, 0) -
                                                                               torch.roll(v, 1, 0))

        db, D = div(q[3], q[4]), n * q[:3]
        dd = div(D[0], D[1])
        return [float((q * q).sum() / (c["Nx"] * c["Ny"])), float((db * db).sum()), float(db.abs().max()),
                float((q[3:] ** 2).sum(0).max().sqrt()), float((dd * dd).sum()), float(dd.abs().max()),
                float((D * D).sum(0).max().sqrt()), None]
    if kind == "batch":
        out = []
        for n, steps, pol, x0, sigma in _batch_inputs(c, seed):
            Ny, Nx = n.shape[1:]
            d = _grid(Nx, Ny)[0] - x0
            d = d - Nx * torch.floor(d / Nx + 0.5)
            g = torch.exp(-d * d / (2.0 * sigma * sigma)).float().double().expand(Ny, Nx)
            q = torch.zeros(6, Ny, Nx, dtype=torch.float64, device=DEV)
            e, b, s = (2, 4, -1.0) if pol == "Ez" else (1, 5, 1.0)
            q[e], q[b] = g, s * g
            out.append(_advance(n, q, 0.05, steps, True, False, "TM" if pol == "Ez" else "TE"))
        return out
    q, n, t = (v.double() for v in _net_inputs(c, seed))
    flat = torch.from_numpy(np.asarray(_params(), dtype=np.float64)).to(DEV)
    flat.requires_grad_(kind == "train")
    params = [(flat[w].view(shape), flat[b]) for w, shape, b in surrogate.param_slices()]
    if kind == "forward":
        return q + _network(q, n, params) / 16.0
    dq = t - q
    grad, num, den = torch.zeros_like(flat), 0.0, float((dq * dq).sum())
    for i in range(c["nimg"]):
        part = ((_network(q[i:i + 1], n[i:i + 1], params) / 16.0 - dq[i:i + 1]) ** 2).sum()
        grad += torch.autograd.grad(part, flat, retain_graph=True)[0]
        num += float(part)
        del part
    return [num / den, (grad / den)]
