"""What this library is asked to do, as cases that can be timed.

Each case is one piece of work that a program using the library does through
its public entry points: a persistence diagram, a whole simplification, a
differentiable loss with its gradient, a batch of fields, the warm-start
network's inference and its gradients.  The fields are the seeded kinds of
``paper_2407_12399_gb300.synthetic`` (Gaussian mixtures with uniform noise,
filament tubes with lattice-gradient noise, the mean of both), generated here
on the GPU so that many of them can be made quickly.

    listed()             the named cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  the inputs and the handles a program keeps
    run(state)           one pass through the public entry points
    work(case)           bytes and operations a pass cannot do without
    exact(case, seed)    the network's outputs in 64 bits
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch

import paper_2407_12399_gb300 as tsf
from paper_2407_12399_gb300 import autograd as tsf_autograd

_WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(tsf.__file__)), "unet_warm_start.npy")

# axes of the fields of a batch
BATCH_DIMS = (48, 64, 96, 128)


def listed():
    return [
        # A diagram of a small field: the interactive or inner-loop call, where
        # launches, read-backs and allocations count.
        {"name": "diagram_mixture_32", "kind": "diagram", "gen": "mixture", "lz": 32, "ly": 32, "lx": 32, "bumps": 8,
         "levels": 0},
        # 8-bit scanner data on an odd grid: many equal values, so plateaus and
        # pairs of zero persistence, and no axis a multiple of a tile.
        {"name": "diagram_8bit_97x61x130", "kind": "diagram", "gen": "mixture", "lz": 97, "ly": 61, "lx": 130,
         "bumps": 24, "levels": 256},
        # A diagram of a full-size data set rich in saddle-saddle pairs.
        {"name": "diagram_filament_128", "kind": "diagram", "gen": "filament", "lz": 128, "ly": 128, "lx": 128,
         "bumps": 64, "levels": 0},
        # Whole simplifications: threshold, iterations to 1 % of the loss, the
        # simplified field.  Small field; full-size filaments; the 256^3 field
        # of the headline; an odd grid; and the handle-cutting mode (alpha_d =
        # 0), whose many iterations each change few vertices.
        {"name": "simplify_mixture_32", "kind": "simplify", "gen": "mixture", "lz": 32, "ly": 32, "lx": 32, "bumps": 8,
         "tau": 0.1, "alpha_b": 0.5, "alpha_d": 0.5, "max_iters": 1000},
        {"name": "simplify_filament_128", "kind": "simplify", "gen": "filament", "lz": 128, "ly": 128, "lx": 128,
         "bumps": 64, "tau": 0.05, "alpha_b": 0.5, "alpha_d": 0.5, "max_iters": 1000},
        {"name": "simplify_both_256", "kind": "simplify", "gen": "both", "lz": 256, "ly": 256, "lx": 256, "bumps": 64,
         "tau": 0.05, "alpha_b": 0.5, "alpha_d": 0.5, "max_iters": 1000},
        {"name": "cut_filament_96", "kind": "simplify", "gen": "filament", "lz": 96, "ly": 96, "lx": 96, "bumps": 48,
         "tau": 0.1, "alpha_b": 0.5, "alpha_d": 0.0, "max_iters": 100},
        # The topological loss as a term of an optimisation: forward and
        # backward at two successive iterates.
        {"name": "loss_mixture_96", "kind": "loss", "gen": "mixture", "lz": 96, "ly": 96, "lx": 96, "bumps": 32,
         "tau": 0.1},
        # Uneven fields solved together, matched by the auction: thresholds and
        # the first (largest) iteration of every field.
        {"name": "batch_uneven_12", "kind": "batch", "n": 12, "shape_seed": 2},
        # The warm-start network: inference on an odd grid and on the headline
        # grid, and the training gradients at the training size.
        {"name": "unet_forward_100x76x52", "kind": "unet_forward", "gen": "mixture", "lz": 100, "ly": 76, "lx": 52,
         "bumps": 16, "tau": 0.05},
        {"name": "unet_forward_256", "kind": "unet_forward", "gen": "both", "lz": 256, "ly": 256, "lx": 256,
         "bumps": 64, "tau": 0.05},
        {"name": "unet_gradients_64", "kind": "unet_gradients", "gen": "filament", "lz": 64, "ly": 64, "lx": 64,
         "bumps": 8, "tau": 0.05},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _axes(rng, lo, hi, cap, multiple=1):
    """Three axes in [lo, hi] with at most cap vertices."""
    while True:
        a = [max(lo, _log_int(rng, lo, hi) // multiple * multiple) for _ in range(3)]
        if a[0] * a[1] * a[2] <= cap:
            return {"lz": a[0], "ly": a[1], "lx": a[2]}


def draw(rng):
    kind = rng.choice(["diagram", "simplify", "loss", "batch", "unet_forward", "unet_gradients"])
    c = {"kind": kind}
    if kind == "batch":
        c["n"] = rng.randint(2, 12)
        c["shape_seed"] = rng.randint(0, 1 << 30)
        return c
    if kind == "diagram":
        c.update(_axes(rng, 12, 160, 128 ** 3))
        c["gen"] = rng.choice(["mixture", "filament", "both"])
        c["bumps"] = rng.randint(4, 64)
        c["levels"] = rng.choice([0, 0, 256, 4096])
    elif kind == "simplify":
        c.update(_axes(rng, 16, 144, 112 ** 3))
        c["gen"] = rng.choice(["mixture", "filament", "both"])
        c["bumps"] = rng.randint(4, 64)
        c["tau"] = round(rng.uniform(0.07, 0.2), 3)
        c["alpha_b"], c["alpha_d"] = rng.choice([(0.5, 0.5), (0.5, 0.5), (0.5, 0.0), (0.0, 0.5)])
        c["max_iters"] = 40
    elif kind == "loss":
        c.update(_axes(rng, 16, 128, 96 ** 3))
        c["gen"] = "mixture"
        c["bumps"] = rng.randint(4, 32)
        c["tau"] = round(rng.uniform(0.07, 0.2), 3)
    else:
        big = kind == "unet_forward"
        c.update(_axes(rng, 8, 256 if big else 96, 224 ** 3 if big else 72 ** 3, multiple=4))
        c["gen"] = rng.choice(["mixture", "filament"])
        c["bumps"] = rng.randint(4, 16)
        c["tau"] = round(rng.uniform(0.02, 0.2), 3)
    return c


# --- fields, on the GPU -------------------------------------------------------

def _coords(shape, device):
    return [torch.linspace(0.0, 1.0, n, device=device).reshape([-1 if i == k else 1 for i in range(3)])
            for k, n in enumerate(shape)]


def _normalise(f):
    lo, hi = f.min(), f.max()
    return ((f - lo) / (hi - lo)).contiguous()


def _noise(shape, seed, device):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed))
    return torch.rand(shape, generator=g, device=device)


def _mixture(shape, bumps, rng, device, noise=0.05):
    """Sum of isotropic Gaussians plus uniform noise of `noise` x its range."""
    c = rng.uniform(0.0, 1.0, (bumps, 3))
    s = rng.uniform(0.05, 0.15, bumps)
    a = rng.uniform(0.5, 1.0, bumps)
    z, y, x = _coords(shape, device)
    f = torch.zeros(shape, device=device)
    for k in range(bumps):
        e = [torch.exp(-(t - float(c[k, i])) ** 2 / (2.0 * float(s[k]) ** 2)) for i, t in enumerate((x, y, z))]
        f += float(a[k]) * (e[2] * e[1]) * e[0]
    if noise > 0:
        f += (f.max() - f.min()) * noise * _noise(shape, rng.integers(0, 1 << 31), device)
    return _normalise(f)


def _gradient_noise(shape, rng, device, octaves=4, base=4):
    """Lattice-gradient noise, frequency x2 and amplitude x1/2 per octave."""
    out = torch.zeros(shape, device=device)
    z, y, x = _coords(shape, device)
    for o in range(octaves):
        freq = base << o
        g = rng.normal(size=(freq + 1, freq + 1, freq + 1, 3))
        g /= np.linalg.norm(g, axis=-1, keepdims=True)
        g = torch.from_numpy(g.astype(np.float32)).to(device)
        cell, t, w = [], [], []
        for p in (x * freq, y * freq, z * freq):
            i = p.floor().clamp(max=freq - 1)
            cell.append(i.long())
            t.append(p - i)
            w.append(t[-1] ** 3 * (t[-1] * (t[-1] * 6.0 - 15.0) + 10.0))
        for cz in (0, 1):
            for cy in (0, 1):
                for cx in (0, 1):
                    at = g[cell[0] + cx, cell[1] + cy, cell[2] + cz]
                    dot = at[..., 0] * (t[0] - cx) + at[..., 1] * (t[1] - cy) + at[..., 2] * (t[2] - cz)
                    k = [w[i] if s else 1 - w[i] for i, s in enumerate((cx, cy, cz))]
                    out += 0.5 ** o * (k[0] * k[1] * k[2]) * dot
    return out


def _filament(shape, loops, rng, device, segs=8):
    """Negative distance to closed polygonal tubes, blurred by one voxel, plus
    lattice-gradient noise of a tenth of the range."""
    centre = rng.uniform(0.15, 0.85, (loops, 3))
    radius = rng.uniform(0.04, 0.15, loops)
    normal = rng.normal(size=(loops, 3))
    jit = rng.uniform(-1, 1, (3, loops, segs))
    z, y, x = _coords(shape, device)
    d2 = torch.full(shape, 1e9, device=device)
    for i in range(loops):
        n = normal[i] / np.linalg.norm(normal[i])
        u = np.cross(n, [1.0, 0.0, 0.0] if abs(n[0]) < 0.9 else [0.0, 1.0, 0.0])
        u /= np.linalg.norm(u)
        v = np.cross(n, u)
        th = 2 * np.pi * (np.arange(segs) + 0.25 * jit[0, i]) / segs
        r = radius[i] * (1.0 + 0.3 * jit[1, i])
        p = (centre[i] + r[:, None] * (np.cos(th)[:, None] * u + np.sin(th)[:, None] * v)
             + (0.2 * radius[i] * jit[2, i])[:, None] * n)
        for a, b in zip(p, np.roll(p, -1, axis=0)):
            ab = b - a
            ax, ay, az = x - float(a[0]), y - float(a[1]), z - float(a[2])
            q = 1.0 / max(float(ab @ ab), 1e-30)
            t = ((az * float(ab[2] * q) + ay * float(ab[1] * q)) + ax * float(ab[0] * q)).clamp_(0.0, 1.0)
            e = (ax - t * float(ab[0])).square_()
            e += (ay - t * float(ab[1])).square_()
            e += (az - t * float(ab[2])).square_()
            torch.minimum(d2, e, out=d2)
    f = 0.02 - d2.sqrt_()
    k = np.exp(-0.5 * np.arange(-3, 4) ** 2)
    k /= k.sum()
    for axis in range(3):
        n = shape[axis]
        idx = torch.arange(n, device=device)
        f = sum(float(k[j + 3]) * f.index_select(axis, (idx + j).clamp(0, n - 1)) for j in range(-3, 4))
    g = _gradient_noise(shape, rng, device)
    return _normalise(f + g * (0.1 * (f.max() - f.min()) / (g.max() - g.min())))


def _field(gen, shape, bumps, rng, device, levels=0):
    if gen == "mixture":
        f = _mixture(shape, bumps, rng, device)
    elif gen == "filament":
        f = _filament(shape, bumps, rng, device)
    else:  # the mean of both, with uniform noise on top
        f = 0.5 * (_mixture(shape, bumps, rng, device, 0.0) + _filament(shape, bumps, rng, device))
        f = _normalise(f + 0.05 * _noise(shape, rng.integers(0, 1 << 31), device))
    if levels:
        f = torch.round(f * (levels - 1)) / (levels - 1)
    return f


def _shape(case):
    return (case["lz"], case["ly"], case["lx"])


def _case_field(case, seed, device="cuda"):
    return _field(case["gen"], _shape(case), case["bumps"], np.random.default_rng([seed, 17]), device,
                  case.get("levels", 0))


def _batch_shapes(case):
    rng = np.random.default_rng([case["shape_seed"], 29])
    return [tuple(int(d) for d in rng.choice(BATCH_DIMS, 3)) for _ in range(case["n"])]


def _unet_pair(case, seed):
    """(f, g): a training input and a stand-in for its simplified field, f
    with its small peaks cut down to their surroundings."""
    f = _case_field(case, seed)
    g = f
    for axis in range(3):
        n = f.shape[axis]
        idx = torch.arange(n, device=f.device)
        g = 0.5 * g + 0.25 * (g.index_select(axis, (idx + 1).clamp(max=n - 1)) +
                              g.index_select(axis, (idx - 1).clamp(min=0)))
    return f, torch.minimum(f, 0.9 * g).contiguous()


# --- preparation --------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "batch":
        rng = np.random.default_rng([seed, 31])
        fields = [_field("mixture", sh, 16, rng, "cuda") for sh in _batch_shapes(case)]
        s["fields"] = fields
        s["out"] = [torch.empty_like(f) for f in fields]
        s["tau"] = rng.uniform(0.07, 0.2, len(fields)).astype(np.float32)
        torch.cuda.synchronize()
        s["batch"] = tsf.Batch(fields)
    elif kind == "loss":
        f = _case_field(case, seed)
        s["field"] = tsf.Field(f)
        s["field"].set_threshold(case["tau"])
        s["iterates"] = [(f + 0.01 * (_noise(f.shape, 2 * seed + k, "cuda") - 0.5)).requires_grad_(True)
                         for k in (0, 1)]
    elif kind == "unet_forward":
        s["f"] = _case_field(case, seed)
        s["net"] = tsf.UNet(np.load(_WEIGHTS))
    elif kind == "unet_gradients":
        f, g = _unet_pair(case, seed)
        s["f"], s["g"] = f.cpu().numpy(), g.cpu().numpy()  # UNet.gradients takes host arrays
        s["net"] = tsf.UNet(np.load(_WEIGHTS))
    else:
        s["f"] = _case_field(case, seed)
        s["field"] = tsf.Field(s["f"])
        if kind == "diagram":  # room for a point per two vertices
            s["out"] = np.zeros(s["f"].numel() // 2 + 64, tsf.PAIR_DTYPE)
        else:
            s["out"] = torch.empty_like(s["f"])
    torch.cuda.synchronize()
    return s


# --- one pass -----------------------------------------------------------------

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "diagram":
        tsf.tsf_set_field(state["field"]._h, state["f"].data_ptr(), 1)
        status, n = tsf.tsf_compute_diagram(state["field"]._h, state["out"].ctypes.data, len(state["out"]))
        if status != tsf.TSF_OK:
            raise tsf.TsfError(status, "tsf_compute_diagram")
        return {"points": n, "pairs": state["out"].view(np.uint8)}
    if kind == "simplify":
        fld = state["field"]
        tsf.tsf_set_field(fld._h, state["f"].data_ptr(), 1)
        fld.set_threshold(case["tau"])
        p = tsf.params(alpha_b=case["alpha_b"], alpha_d=case["alpha_d"], stop_s=0.01, max_iters=case["max_iters"])
        st = tsf.tsf_simplify(fld._h, p, state["out"].data_ptr(), 1)
        return {"values": state["out"], "loss0": st.loss0, "loss": st.loss, "iters": st.iters,
                "points": st.n_points, "uncancelled": st.n_uncancelled}
    if kind == "loss":
        out = []
        for f in state["iterates"]:
            f.grad = None
            loss = tsf_autograd.topological_loss(f, state["field"])
            loss.backward()
            out += [loss.detach(), f.grad]
        return out
    if kind == "batch":
        b = state["batch"]
        for m, f in zip(b.fields, state["fields"]):
            tsf.tsf_set_field(m._h, f.data_ptr(), 1)
        b.set_thresholds(state["tau"])
        stats = b.step(assignment_precision=0.01)
        for m, o in zip(b.fields, state["out"]):
            tsf.tsf_get_field(m._h, o.data_ptr(), 1)
        return {"values": state["out"], "loss": [t["loss"] for t in stats], "points": [t["n_points"] for t in stats]}
    if kind == "unet_forward":
        return state["net"].forward(state["f"], case["tau"])
    loss, grad = state["net"].gradients(state["f"], state["g"], case["tau"])
    return {"loss": loss, "grad": grad}


# --- what a pass cannot do without ----------------------------------------------

def _unet_macs(v):
    """Multiply-adds of one forward pass on v voxels (3x3x3 convolutions, the
    half grid at v/8, the quarter grid at v/64, and the head)."""
    full = 2 * 16 + 16 * 16 + 48 * 16 + 16 * 16
    half = 16 * 32 + 32 * 32 + 96 * 32 + 32 * 32
    quarter = 32 * 64 + 64 * 64
    return v * (27 * (full + half / 8 + quarter / 64) + 16)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        v = sum(a * b * c for a, b, c in _batch_shapes(case))
        return {"bytes": 8.0 * v, "flops": 28.0 * v}
    v = case["lz"] * case["ly"] * case["lx"]
    if kind == "unet_forward":
        return {"bytes": 8.0 * v, "flops": 2.0 * _unet_macs(v)}
    if kind == "unet_gradients":
        # data gradients of all but the first layer, weight gradients of all
        return {"bytes": 8.0 * v + 4.0 * tsf.TSF_UNET_NPARAMS, "flops": 6.0 * _unet_macs(v)}
    if kind == "loss":
        # two evaluations: values in, the fp32 gradient out; 14 comparisons per vertex
        return {"bytes": 2 * 8.0 * v, "flops": 2 * 14.0 * v}
    # values in; the diagram (about a twentieth of the vertices on noisy
    # fields, 40 bytes a point) or the simplified values out.  At least two
    # diagrams per simplification.
    if kind == "diagram":
        return {"bytes": 6.0 * v, "flops": 14.0 * v}
    return {"bytes": 8.0 * v, "flops": 28.0 * v}


# --- the network in 64 bits -----------------------------------------------------

def _conv64(x, w, b):
    """3x3x3 cross-correlation with zero padding; x (C, Z, Y, X), w (O, C, 3, 3, 3)."""
    c, nz, ny, nx = x.shape
    xp = torch.nn.functional.pad(x, (1, 1, 1, 1, 1, 1))
    y = b.reshape(-1, 1).expand(-1, nz * ny * nx)
    for dz in range(3):
        for dy in range(3):
            for dx in range(3):
                win = xp[:, dz:dz + nz, dy:dy + ny, dx:dx + nx].reshape(c, -1)
                y = y + w[:, :, dz, dy, dx] @ win
    return y.reshape(-1, nz, ny, nx)


def _unet64(p, f, tau):
    def layer(name, x):
        return torch.relu(_conv64(x, p[name + ".w"], p[name + ".b"]))

    def pool(x):
        c, z, y, w = x.shape
        return x.reshape(c, z // 2, 2, y // 2, 2, w // 2, 2).mean(dim=(2, 4, 6))

    def up(x):
        return x.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)

    x = torch.stack([f, torch.full_like(f, tau)])
    e1 = layer("e1b", layer("e1a", x))
    e2 = layer("e2b", layer("e2a", pool(e1)))
    e3 = layer("e3b", layer("e3a", pool(e2)))
    d2 = layer("d2b", layer("d2a", torch.cat([up(e3), e2])))
    d1 = layer("d1b", layer("d1a", torch.cat([up(d2), e1])))
    return f + torch.einsum("c,czyx->zyx", p["head.w"][0], d1) + p["head.b"][0]


def exact(case, seed):
    """The network's outputs from its fp32 parameters, in float64.  The other
    cases' outputs are combinatorial, or follow from such."""
    if case["kind"] not in ("unet_forward", "unet_gradients"):
        return None
    # layer by layer in the parameter order that tsf.h states
    chans = [("e1a", 16, 2), ("e1b", 16, 16), ("e2a", 32, 16), ("e2b", 32, 32), ("e3a", 64, 32), ("e3b", 64, 64),
             ("d2a", 32, 96), ("d2b", 32, 32), ("d1a", 16, 48), ("d1b", 16, 16)]
    specs = [(n, (o, i, 3, 3, 3), o) for n, o, i in chans] + [("head", (1, 16), 1)]
    flat = torch.from_numpy(np.load(_WEIGHTS).astype(np.float64)).cuda()
    grads = case["kind"] == "unet_gradients"
    flat.requires_grad_(grads)
    p, o = {}, 0
    for name, shape, nb in specs:
        k = math.prod(shape)
        p[name + ".w"] = flat[o:o + k].reshape(shape)
        p[name + ".b"] = flat[o + k:o + k + nb]
        o += k + nb
    if not grads:
        with torch.no_grad():
            return _unet64(p, _case_field(case, seed).double(), case["tau"])
    f, g = (t.double() for t in _unet_pair(case, seed))
    loss = (_unet64(p, f, case["tau"]) - g).square().mean()
    loss.backward()
    return {"loss": float(loss), "grad": flat.grad.cpu().numpy()}
