"""Performance cases of the filament-fluid step: what users of this framework have it do.

A case is a dict of plain values; its "kind" is the call that a program makes:

  step    one resident world advanced by `steps` time steps, then its beads
          (and with `fluid` its populations) read back on the device
  batch   `worlds` uneven worlds advanced together, then every world's beads
  serve   `worlds` rollout requests submitted to a continuous-batching server
          and waited for (the worlds are created, stepped, reduced and freed
          inside the call, as in a search loop)
  grad    one iteration of the folding optimisation: new rest angles, the
          recorded rollout, the loss, the reverse sweep with every gradient

Grids are multiples of 8 cells a side, as the library requires; filaments have
`bmin` to `bmax` beads.  Inputs are drawn from the seed alone.  exact() is the
same physics in 64-bit torch operations (autograd for the gradients), written
from the model's equations.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2607_02954_gb300 import Server, World, step_batched, synth
from paper_2607_02954_gb300 import _lib as L
from paper_2607_02954_gb300.world import stream_handle

# Every option of a world with its default; a case names the ones it changes.
OPTIONS = dict(nu=0.1, sigma=1.0, n_pbd=4, order=0, layers=1, ib=0, mdf=0, observe=False)


def case_of(kind, **kw):
    return {"kind": kind, **OPTIONS, **kw}


def listed():
    return [
        # An interactive loop: a small tank, one step, the beads read back.
        case_of("step", name="tick_64", H=64, W=64, fil=6, bmin=8, bmax=64, steps=1, fluid=False),
        # The repository's small world (16 filaments of 32 beads on 128^2), a burst of steps between two looks at it.
        case_of("step", name="swim_128", H=128, W=128, fil=16, bmin=32, bmax=32, steps=100, fluid=False),
        # An odd grid with ragged last tiles, filaments on both sides of 64 beads, the widest filter, red-black passes.
        case_of("step", name="mixed_200x328", H=200, W=328, fil=60, bmin=2, bmax=300, steps=48, fluid=True,
                sigma=2.0, order=1),
        # The repository's 512^2 world of 4096 filaments of 64 beads (one bead per cell).
        case_of("step", name="crowd_512", H=512, W=512, fil=4096, bmin=64, bmax=64, steps=32, fluid=False),
        # The scalability shape: 2^18 beads on 256^2, four per cell.
        case_of("step", name="dense_256", H=256, W=256, fil=4096, bmin=64, bmax=64, steps=24, fluid=False),
        # The headline point of the particle-count sweep: 2^22 beads on 4096^2.
        case_of("step", name="sweep_4096", H=4096, W=4096, fil=65536, bmin=64, bmax=64, steps=16, fluid=True),
        # What the search experiments read: a rest-length drive, an energy field, the behaviour descriptors.
        case_of("step", name="observed_1000x1480", H=1000, W=1480, fil=8000, bmin=24, bmax=64, steps=16, fluid=False,
                observe=True),
        # Direct forcing with four passes, the coupling for stiff swimmers.
        case_of("step", name="forced_1024", H=1024, W=1024, fil=4096, bmin=64, bmax=64, steps=16, fluid=False,
                ib=1, mdf=4),
        # Uneven worlds of 64 to 256 cells a side stepped together.
        case_of("batch", name="batch_256", worlds=256, side_min=64, side_max=256, fil=64, bmin=8, bmax=64, steps=48),
        # A search generation through the server, with the observables it ranks by.
        case_of("serve", name="serve_96", worlds=96, side_min=64, side_max=256, fil=64, bmin=8, bmax=64, steps=80,
                tick=10, observe=True),
        # The folding optimisation on 256^2, 64 filaments of 48 beads, checkpointed.
        case_of("grad", name="fold_256", H=256, W=256, fil=64, bmin=48, bmax=48, steps=200, every=50, stored=False,
                loss="polyline"),
        # A larger folding world of two-layer filaments against an image, every step stored.
        case_of("grad", name="fold_stored_488x640", H=488, W=640, fil=300, bmin=16, bmax=64, steps=32, every=32,
                stored=True, loss="splat", layers=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above."""
    kind = rng.choice(["step"] * 6 + ["batch", "serve"] + ["grad"] * 3)
    opt = {}
    if rng.random() < 0.5:
        opt["sigma"] = rng.choice([0.5, 0.75, 1.25, 1.5, 2.0])
    if rng.random() < 0.3:
        opt["order"] = 1
    if rng.random() < 0.4:
        opt["n_pbd"] = rng.choice([1, 2, 3, 6, 8])
    if rng.random() < 0.5:
        opt["nu"] = round(rng.uniform(0.06, 0.4), 3)
    if kind in ("batch", "serve"):
        hi = rng.choice([64, 128, 256])
        bmax = rng.choice([24, 64, 64, 100])
        c = case_of(kind, worlds=_log_int(rng, 4, 256 if kind == "batch" else 96), side_min=rng.choice([32, 64]),
                    side_max=hi, fil=_log_int(rng, 4, 64), bmin=rng.choice([2, 8]), bmax=bmax,
                    steps=_log_int(rng, 12, 64), **opt)
        if kind == "serve":
            c["tick"] = rng.choice([5, 10, 20])
            c["observe"] = rng.random() < 0.7
        return c
    # grid sides over the whole range, odd multiples of 8 and unequal sides among them
    top = 4096 if kind == "step" else 640
    H = 8 * _log_int(rng, 6, top // 8)
    W = 8 * max(6, min(top // 8, int(round(H / 8 * rng.uniform(0.5, 2.0)))))
    bmax = rng.choice([16, 48, 64, 64, 64, 120, 300]) if kind == "step" else rng.choice([24, 48, 64, 90])
    bmax = min(bmax, W - 8)
    bmin = rng.choice([2, 8, bmax])
    bmin = min(bmin, bmax)
    mean = (bmin + bmax) / 2
    per_cell = math.exp(rng.uniform(math.log(0.02), math.log(1.0 if kind == "step" else 0.08)))
    fil = max(1, min(int(H * W * per_cell / mean), 65536))
    extra = rng.choice(["", "", "layers", "forced", "observe"])
    if extra == "layers":
        opt["layers"] = 2
    elif extra == "forced":
        opt["ib"], opt["mdf"] = 1, rng.choice([1, 2, 3, 4])
    elif extra == "observe" and kind == "step":
        opt["observe"] = True
    # steps so that a pass costs no more than the largest listed one
    most = 2.0e8 / (H * W * (4 if extra in ("layers", "forced") else 1) + 4.0 * fil * mean)
    if kind == "step":
        steps = max(1, min(_log_int(rng, 1, 100), int(most)))
        return case_of("step", H=H, W=W, fil=fil, bmin=bmin, bmax=bmax, steps=steps, fluid=rng.random() < 0.4, **opt)
    if opt.get("n_pbd", 4) > 4 and bmax > 64:
        opt["n_pbd"] = 4
    steps = max(4, min(_log_int(rng, 8, 200), int(most / 4)))
    return case_of("grad", H=H, W=W, fil=fil, bmin=bmin, bmax=bmax, steps=steps,
                   every=max(1, int(round(steps / rng.choice([1, 2, 4, 5])))), stored=rng.random() < 0.4,
                   loss=rng.choice(["polyline", "splat"]), **opt)


# ---------------------------------------------------------------------------
# Inputs.
# ---------------------------------------------------------------------------
def _spec(rng, H, W, fil, bmin, bmax, case, drive=True):
    """Filaments of bmin..bmax beads (log-uniform, the same ones for every
    seed) on a jittered row lattice of the whole grid, rest angles ~N(0, 0.1)
    and a travelling-wave drive (none for the folding worlds, whose rest angles
    are what is optimised)."""
    sizes = np.random.default_rng(fil)
    B = np.exp(sizes.uniform(math.log(bmin), math.log(bmax), fil)).round().astype(np.int64) if bmin < bmax \
        else np.full(fil, bmin, np.int64)
    slot = min(int(B.max()) + (0 if bmin == bmax and bmax % 8 == 0 else 2), W)
    per_row = max(1, W // slot)
    rows = -(-fil // per_row)
    f = np.arange(fil)
    x0 = (f % per_row) * (W / per_row) + rng.uniform(0.0, 0.5, fil)
    y0 = (f // per_row) * (H / rows) + rng.uniform(0.0, 0.5, fil)
    flip = rng.integers(0, 2, fil)
    off = np.zeros(fil + 1, np.int64)
    off[1:] = np.cumsum(B)
    of = np.repeat(f, B)
    k = np.arange(off[-1]) - off[of]
    along = np.where(flip[of] == 1, B[of] - 1 - k, k)
    x = np.mod(x0[of] + along, W).astype(np.float32)
    y = np.mod(y0[of], H).astype(np.float32)
    x[x >= W] = 0.0
    y[y >= H] = 0.0
    theta = np.repeat(flip * math.pi, B - 1).astype(np.float32)
    J = int((B - 2).sum())
    jf = np.repeat(f, B - 2)
    local = np.arange(J) - np.concatenate([[0], np.cumsum(B - 2)])[jf]
    theta0 = rng.normal(0.0, 0.1, J).astype(np.float32)
    amp = np.full(J, 0.3 if drive else 0.0, np.float32)
    freq = np.full(J, 1.0 / 200.0 if drive else 0.0, np.float32)
    phase = np.mod(rng.uniform(0, 1, fil)[jf] - local / 16.0, 1.0).astype(np.float32)
    # the default repulsion is for at most about one bead per cell
    k_rep = 0.5 * min(1.0, 0.5 * H * W / max(1, int(off[-1])))
    p = synth.Params(nu=case["nu"], sigma=case["sigma"], n_pbd=case["n_pbd"], pbd_order=case["order"],
                     layers=case["layers"], ib=case["ib"], mdf_iters=case["mdf"], k_rep=k_rep)
    s = synth.WorldSpec(H=H, W=W, fil_off=off.astype(np.int32), x=x, y=y, theta=theta,
                        L_rest=np.ones(int(off[-1]) - fil, np.float32), theta0=theta0, drive_amp=amp, drive_freq=freq,
                        drive_phase=phase, params=p)
    if case["observe"]:
        E = s.E
        s.len_amp = rng.uniform(0.0, 0.2, E).astype(np.float32)
        s.len_freq = (1.0 / rng.uniform(50.0, 400.0, E)).astype(np.float32)
        s.len_phase = rng.uniform(0.0, 1.0, E).astype(np.float32)
        ys, xs = np.arange(H)[:, None], np.arange(W)[None, :]
        en = np.zeros((H, W), np.float32)
        for _ in range(4):   # periodic Gaussian-like packets (separable)
            cx, cy, wd, a = rng.uniform(0, W), rng.uniform(0, H), rng.uniform(4.0, 12.0), rng.uniform(0.2, 1.0)
            dx, dy = xs - cx, ys - cy
            dx, dy = dx - W * np.round(dx / W), dy - H * np.round(dy / H)
            en += (a * np.exp(-dy * dy / (2 * wd * wd)) * np.exp(-dx * dx / (2 * wd * wd))).astype(np.float32)
        s.energy = en
        s.observe = True
    return s


def _specs(case, seed):
    """The worlds of a batch or a generation: sides of a power of two from
    side_min to side_max, 1 to `fil` filaments (log-uniform); the sizes are
    the same for every seed."""
    rng, sizes = np.random.default_rng(seed), np.random.default_rng(case["worlds"])
    sides = [s for s in (32, 64, 128, 256) if case["side_min"] <= s <= case["side_max"]] or [case["side_max"]]
    out = []
    for _ in range(case["worlds"]):
        side = int(sizes.choice(sides))
        bmax = min(case["bmax"], side - 4)
        most = max(1, min(case["fil"], side * side // (4 * bmax)))
        fil = int(round(math.exp(sizes.uniform(0.0, math.log(most + 0.49)))))
        out.append(_spec(rng, side, side, max(1, fil), min(case["bmin"], bmax), bmax, case))
    return out


def _one(case, seed):
    rng = np.random.default_rng(seed)
    return _spec(rng, case["H"], case["W"], case["fil"], case["bmin"], case["bmax"], case, drive=case["kind"] == "step")


def _target(case, seed):
    """The folding target: a polyline of 16 vertices, or a 128 x 128 image of two soft strokes."""
    rng = np.random.default_rng(seed + 1)
    H, W = case["H"], case["W"]
    if case["loss"] == "polyline":
        return np.stack([rng.uniform(0, W, 16), rng.uniform(0, H, 16)], 1).astype(np.float32)
    R = 128
    c = np.arange(R) + 0.5
    img = np.zeros((R, R))
    for _ in range(2):
        P = rng.uniform(0.2 * R, 0.8 * R, (3, 2))
        for t in np.linspace(0.0, 1.0, 48):
            q = (1 - t) ** 2 * P[0] + 2 * (1 - t) * t * P[1] + t * t * P[2]
            img = np.maximum(img, np.exp(-(c - q[1]) ** 2 / 12.5)[:, None] * np.exp(-(c - q[0]) ** 2 / 12.5)[None, :])
    return img.astype(np.float32)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        return {"case": case, "server": Server(max_slots=1024, steps_per_tick=case["tick"]), "specs": _specs(case, seed)}
    if kind == "batch":
        return {"case": case, "worlds": [World(s) for s in _specs(case, seed)]}
    w = World(_one(case, seed))
    st = {"case": case, "world": w}
    if kind == "grad":
        st["theta0"] = torch.from_numpy(w.spec.theta0).cuda()
        st["target"] = _target(case, seed)
        if case["loss"] == "splat":
            st["target"] = torch.from_numpy(st["target"]).cuda()
        st["recorded"] = False
    return st


# ---------------------------------------------------------------------------
# The measured pass.
# ---------------------------------------------------------------------------
def _read_fluid(w):
    """The populations (minus the rest weights) into device memory, as mc_world_get_state gives them."""
    out = torch.empty((9, w.spec.H, w.spec.W), device="cuda")
    L.check(L.load().mc_world_get_state(w.handle, None, None, None, None, ctypes.c_void_p(out.data_ptr()),
                                        L.MC_MEM_DEVICE, stream_handle()))
    return out


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        w = state["world"]
        w.step(case["steps"])
        out = w.state_device()
        if case["fluid"]:
            out["fluid"] = _read_fluid(w)
        if case["observe"]:
            o = w.observables()
            out["observables"] = np.array([o["e_bend"], o["e_pos"], o["energy"]])
        return out
    if kind == "batch":
        ws = state["worlds"]
        step_batched(ws, case["steps"])
        each = [w.state_device() for w in ws]
        return {k: torch.cat([e[k] for e in each]) for k in ("x", "y", "theta", "disp")}
    if kind == "serve":
        srv = state["server"]
        tickets = [srv.submit(s, case["steps"]) for s in state["specs"]]
        res = [srv.wait(t) for t in tickets]
        return {"com_disp": np.array([r["com_disp"] for r in res]),
                "observables": np.array([[r["e_bend"], r["e_pos"], r["energy"]] for r in res]),
                "status": np.array([r["status"] for r in res], np.int64)}
    w = state["world"]
    if state["recorded"]:
        w.rollout_rewind()
    w.set_rest(theta0=state["theta0"])
    w.rollout_forward(case["steps"], case["every"], stored=case["stored"])
    state["recorded"] = True
    loss, gx, gy = w.loss_polyline(state["target"]) if case["loss"] == "polyline" else w.loss_splat(state["target"])
    g = w.rollout_backward_params(gx, gy)
    return {"loss": loss, "gx": gx, "gy": gy, "theta0": g["theta0"], "L_rest": g["L_rest"], "k": g["k"]}


# ---------------------------------------------------------------------------
# What a pass cannot do without.
# ---------------------------------------------------------------------------
def _sizes(case):
    """(cells, beads) of all worlds, as expected from the distributions."""
    mean = case["bmin"] if case["bmin"] == case["bmax"] else \
        (case["bmax"] - case["bmin"]) / math.log(case["bmax"] / case["bmin"])
    if case["kind"] in ("step", "grad"):
        return case["H"] * case["W"], case["fil"] * mean
    sides = [s for s in (32, 64, 128, 256) if case["side_min"] <= s <= case["side_max"]] or [case["side_max"]]
    fil = (case["fil"] - 1) / math.log(case["fil"]) if case["fil"] > 1 else 1
    return case["worlds"] * sum(s * s for s in sides) / len(sides), case["worlds"] * fil * mean


def work(case):
    """Each step reads and writes a cell's nine populations and a bead's
    position, displacement and edge angle, and reads its rest length and
    drive; a reversed step reads the step's populations and fields and reads
    and writes their adjoints."""
    cells, beads = _sizes(case)
    n = case["steps"]
    per_cell, per_bead = 72.0, 2 * (16 + 8 + 4) + 4 + 16
    if case["observe"]:
        per_cell += 4.0
        per_bead += 12.0
    b = n * (per_cell * cells + per_bead * beads)
    f = n * (190.0 * cells + (260.0 + 60.0 * case["n_pbd"] + 140.0 * case["mdf"]) * beads)
    if case["kind"] == "grad":
        b += n * ((36.0 + 8.0 + 72.0) * cells + (36.0 + 2 * 12.0) * beads)
        f *= 3.5
    if case.get("fluid"):
        b += 72.0 * cells
    b += 28.0 * beads
    return {"bytes": b, "flops": f}


def tolerance(case):
    """About four times the distance of the outputs from the 64-bit result,
    which any other order of the 32-bit operations shows as well: positions,
    angles and displacements were seen 2e-7 to 9e-7 off (a second burst of
    steps starts from the first one's rounding), gradients 9e-6 with the
    polyline and 1.5e-4 with the image, whose bead gradients nearly cancel."""
    if case["kind"] == "grad":
        return {"rel": 4e-5, "max": 4e-3} if case["loss"] == "polyline" else {"rel": 6e-4, "max": 0.06}
    return {"rel": 1e-5, "max": 1e-3}


# ---------------------------------------------------------------------------
# The same pass in 64 bits.
# ---------------------------------------------------------------------------
CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
WT = (4.0 / 9.0,) + (1.0 / 9.0,) * 4 + (1.0 / 36.0,) * 4
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)


def _phi(r):
    """Peskin's 4-point kernel."""
    a = r.abs()
    near, far = a.clamp(max=1.0), a.clamp(min=1.0, max=2.0)
    inner = (3.0 - 2.0 * near + torch.sqrt(1.0 + 4.0 * near - 4.0 * near * near)) / 8.0
    outer = (5.0 - 2.0 * far - torch.sqrt((-7.0 + 12.0 * far - 4.0 * far * far).clamp(min=1e-30))) / 8.0
    return torch.where(a <= 1.0, inner, torch.where(a < 2.0, outer, torch.zeros_like(a)))


class _Exact:
    """Worlds of one grid size side by side: beads concatenated, grids stacked."""

    def __init__(self, specs):
        s0 = specs[0]
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.H, self.W, self.M = s0.H, s0.W, len(specs)
        r = lambda v: float(np.float32(v))
        p = s0.params
        self.p = {k: r(getattr(p, k)) for k in ("nu", "dt", "Lambda", "kappa", "k_bend", "k_stretch", "k_shear",
                                                 "sigma", "orient", "layer_half")}
        self.n_pbd, self.order, self.layers, self.ib, self.mdf = p.n_pbd, p.pbd_order, p.layers, p.ib, p.mdf_iters
        cat = lambda name: self.put(np.concatenate([getattr(s, name) for s in specs]))
        self.X = torch.stack([cat("x"), cat("y")], 1)
        self.th, self.L0, self.th0 = cat("theta"), cat("L_rest"), cat("theta0")
        self.amp, self.freq, self.phase = cat("drive_amp"), cat("drive_freq"), cat("drive_phase")
        self.len = None if s0.len_amp is None else (cat("len_amp"), cat("len_freq"), cat("len_phase"))
        self.energy = None if s0.energy is None else self.put(np.stack([s.energy for s in specs]))
        ws, ea, j1, ep, jp, ew, jw, base, eb = [], [], [], [], [], [], [], 0, 0
        for m, s in enumerate(specs):
            B = np.diff(s.fil_off).astype(np.int64)
            f = np.arange(len(B))
            start = s.fil_off[:-1].astype(np.int64)
            ef = np.repeat(f, B - 1)
            le = np.arange(len(ef)) - (start - f)[ef]
            ea.append(base + start[ef] + le)
            ep.append(le % 2)
            jf = np.repeat(f, B - 2)
            lj = np.arange(len(jf)) - (start - 2 * f)[jf]
            j1.append(eb + (start - f)[jf] + lj)
            jp.append(lj % 2)
            ws.append(np.full(s.N, m))
            ew.append(np.full(s.E, m))
            jw.append(np.full(s.J, m))
            base += s.N
            eb += s.E
        self.w, self.ew, self.jw = self.idx(ws), self.idx(ew), self.idx(jw)
        self.ea, self.j1 = self.idx(ea), self.idx(j1)
        self.ep, self.jp = self.idx(ep), self.idx(jp)
        self.k_rep = self.put(np.array([np.float32(s.params.k_rep) for s in specs]))[self.w]
        self.t = 0
        self.f = self.put(np.array(WT))[None, :, None, None].expand(self.M, 9, self.H, self.W).clone()
        self.D = torch.zeros_like(self.X)
        self.obs = torch.zeros((self.M, 3), dtype=torch.float64, device=self.dev)

    def put(self, a):
        return torch.as_tensor(np.asarray(a, np.float64)).to(self.dev)

    def idx(self, parts):
        return torch.as_tensor(np.concatenate(parts).astype(np.int64)).to(self.dev)

    # -- pieces ---------------------------------------------------------------
    def rest(self, t):
        return self.th0 + self.amp * torch.sin(2 * math.pi * (self.freq * t + self.phase))

    def length(self, t):
        if self.len is None:
            return self.L0
        a, f, p = self.len
        return self.L0 * (1.0 + a * torch.sin(2 * math.pi * (f * t + p)))

    def box(self, d):
        n = torch.tensor([float(self.W), float(self.H)], dtype=torch.float64, device=self.dev)
        return d - n * torch.round(d / n)

    def wrapped(self, X):
        n = torch.tensor([float(self.W), float(self.H)], dtype=torch.float64, device=self.dev)
        Y = X - n * torch.floor(X / n)
        return torch.where(Y >= n, Y - n, Y)

    def stencil(self, X):
        o = torch.arange(-1, 3, device=self.dev)
        b = torch.floor(X).detach()
        cx, cy = b[:, :1] + o, b[:, 1:] + o
        wx, wy = _phi(cx - X[:, :1]), _phi(cy - X[:, 1:])
        ix, iy = torch.remainder(cx.long(), self.W), torch.remainder(cy.long(), self.H)
        i = (self.w[:, None, None] * self.H + iy[:, :, None]) * self.W + ix[:, None, :]
        return i.reshape(-1, 16), (wy[:, :, None] * wx[:, None, :]).reshape(-1, 16)

    def spread(self, st, v):
        i, g = st
        out = torch.zeros(self.M * self.H * self.W, dtype=torch.float64, device=self.dev)
        return out.index_add(0, i.reshape(-1), (g * v[:, None]).reshape(-1)).reshape(self.M, self.H, self.W)

    def gather(self, st, field):
        i, g = st
        return (g * field.reshape(-1)[i]).sum(1)

    def spread2(self, st, v):
        return torch.stack([self.spread(st, v[:, 0]), self.spread(st, v[:, 1])])

    def gather2(self, st, u):
        return torch.stack([self.gather(st, u[0]), self.gather(st, u[1])], 1)

    def blur(self, r):
        R = math.ceil(4.0 * self.p["sigma"])
        m = torch.arange(-R, R + 1, dtype=torch.float64)
        g = torch.exp(-m * m / (2.0 * self.p["sigma"] ** 2))
        g = (g / g.sum()).tolist()
        for d in (2, 1):
            acc = torch.zeros_like(r)
            for k in range(2 * R + 1):
                acc = acc + g[k] * torch.roll(r, k - R, d)
            r = acc
        return r

    def solve(self, X, th, t):
        """The filament solver from positions X: returns the correction and the angles."""
        p, nE = self.p, self.ea.numel()
        rest, Lr = self.rest(t), self.length(t)
        v0 = self.box(X[self.ea + 1] - X[self.ea])
        d = torch.zeros_like(X)
        half = 0.5 * p["k_stretch"]
        for _ in range(self.n_pbd):
            for c in ((0, 1) if self.order else (None,)):
                C = th[self.j1 + 1] - th[self.j1] - rest
                if c is not None:
                    C = C * (self.jp == c)
                C = 0.5 * p["k_bend"] * C
                th = th.index_add(0, self.j1, C).index_add(0, self.j1 + 1, -C) if C.numel() else th
            for c in ((0, 1) if self.order else (None,)):
                v = v0 + d[self.ea + 1] - d[self.ea]
                l = torch.sqrt((v * v).sum(1))
                n = torch.stack([torch.cos(th), torch.sin(th)], 1)
                s = ((l - Lr) / l)[:, None] * v
                dx = half * (s + p["k_shear"] * (v - Lr[:, None] * n - s))
                turn = p["orient"] * half * p["k_shear"] * (n[:, 0] * v[:, 1] - n[:, 1] * v[:, 0]) / Lr
                if c is not None:
                    dx, turn = dx * (self.ep == c)[:, None], turn * (self.ep == c)
                if nE:
                    d = d.index_add(0, self.ea, dx).index_add(0, self.ea + 1, -dx)
                    th = th + turn
        return d, th

    def normals(self, X):
        v = self.box(X[self.ea + 1] - X[self.ea])
        v = v / torch.sqrt((v * v).sum(1, keepdim=True))
        out = torch.zeros_like(X).index_add(0, self.ea, v)
        s = out.index_add(0, self.ea + 1, v)
        n = torch.sqrt((s * s).sum(1, keepdim=True))
        last = torch.ones(X.shape[0], dtype=torch.bool, device=self.dev)
        last[self.ea] = False
        t = torch.where(n >= 1e-3, s / n.clamp(min=1e-30), torch.where(last[:, None], s - out, out))
        return torch.stack([-t[:, 1], t[:, 0]], 1)

    def moments(self, F):
        rho = self.f.sum(1)
        jx = sum(c * self.f[:, i] for i, c in enumerate(CX) if c)
        jy = sum(c * self.f[:, i] for i, c in enumerate(CY) if c)
        return rho, (jx + 0.5 * F[0]) / rho, (jy + 0.5 * F[1]) / rho

    def fluid(self, F):
        """Two-relaxation-time collision with Guo's forcing, then streaming; returns u."""
        tp = 3.0 * self.p["nu"] + 0.5
        tm = 0.5 + self.p["Lambda"] / (tp - 0.5)
        rho, ux, uy = self.moments(F)
        uu, uF = ux * ux + uy * uy, ux * F[0] + uy * F[1]
        new = [None] * 9
        for i in (0, 1, 2, 5, 6):
            o = OPP[i]
            cu, cF = CX[i] * ux + CY[i] * uy, CX[i] * F[0] + CY[i] * F[1]
            ep = WT[i] * rho * (1.0 + 4.5 * cu * cu - 1.5 * uu)
            em = WT[i] * rho * 3.0 * cu
            sp, sm = WT[i] * (9.0 * cu * cF - 3.0 * uF), WT[i] * 3.0 * cF
            fi, fo = self.f[:, i], self.f[:, o]
            even = -(0.5 * (fi + fo) - ep) / tp + (1.0 - 0.5 / tp) * sp
            odd = -(0.5 * (fi - fo) - em) / tm + (1.0 - 0.5 / tm) * sm
            new[i] = torch.roll(fi + even + odd, (CY[i], CX[i]), (1, 2))
            if o != i:
                new[o] = torch.roll(fo + even - odd, (CY[o], CX[o]), (1, 2))
        self.f = torch.stack(new, 1)
        return torch.stack([ux, uy])

    def observe(self, st):
        t = self.t
        if t >= 1:
            self.obs[:, 0].index_add_(0, self.jw, (self.rest(t - 1) - self.rest(t)) ** 2)
            self.obs[:, 1].index_add_(0, self.ew, (self.length(t - 1) - self.length(t)) ** 2)
        if self.energy is not None:
            self.obs[:, 2].index_add_(0, self.w, self.gather(st, self.energy))

    def step(self, observe=False):
        p, X, dt = self.p, self.X, self.p["dt"]
        st = self.stencil(X)
        if observe:
            self.observe(st)
        rb = self.blur(self.spread(st, torch.ones_like(X[:, 0])))
        grad = torch.stack([0.5 * (torch.roll(rb, -1, 2) - torch.roll(rb, 1, 2)),
                            0.5 * (torch.roll(rb, -1, 1) - torch.roll(rb, 1, 1))])
        Fs = -self.k_rep[:, None] * self.gather2(st, grad)
        if self.ib == 1:
            F = self.spread2(st, Fs)
            rho, ux, uy = self.moments(F)
            u = torch.stack([ux, uy])
            drag = self.gather2(st, u)
            d, self.th = self.solve(self.wrapped(X + dt * drag), self.th, self.t)
            U = drag + d / dt
            for _ in range(self.mdf):
                G = self.spread2(st, 2.0 * self.gather(st, rho)[:, None] * (U - self.gather2(st, u)))
                F, u = F + G, u + G / (2.0 * rho)
            self.fluid(F)
        else:
            d, self.th = self.solve(X, self.th, self.t)
            Ft = p["kappa"] / dt * d + Fs
            if self.layers == 2:
                n = p["layer_half"] * self.normals(X)
                pts = [self.stencil(self.wrapped(X + n)), self.stencil(self.wrapped(X - n))]
                u = self.fluid(self.spread2(pts[0], 0.5 * Ft) + self.spread2(pts[1], 0.5 * Ft))
                U = 0.5 * (self.gather2(pts[0], u) + self.gather2(pts[1], u))
            else:
                U = self.gather2(st, self.fluid(self.spread2(st, Ft)))
        self.X, self.D = self.wrapped(X + dt * U), self.D + dt * U
        self.t += 1


def _exact_loss(e, case, X0, target):
    if case["loss"] == "polyline":
        P = X0 + e.D
        v = e.put(target)
        A, AB = v[:-1], v[1:] - v[:-1]
        AP = P[:, None] - A[None]
        t = ((AP * AB).sum(-1) / (AB * AB).sum(-1)).clamp(0.0, 1.0)
        q = AP - t[..., None] * AB
        return (q * q).sum(-1).min(1).values.mean()
    R, K = target.shape[0], 4
    o = torch.arange(-K, K + 1, device=e.dev)
    # the final positions through the displacement, so that its gradient is the loss's gradient
    u = torch.remainder(X0 + e.D, torch.tensor([float(e.W), float(e.H)], dtype=torch.float64, device=e.dev))
    ux, uy = u[:, :1] * R / e.W, u[:, 1:] * R / e.H
    px, py = torch.floor(ux).detach() + o, torch.floor(uy).detach() + o
    gx, gy = torch.exp(-0.5 * (px + 0.5 - ux) ** 2), torch.exp(-0.5 * (py + 0.5 - uy) ** 2)
    i = torch.remainder(py.long(), R)[:, :, None] * R + torch.remainder(px.long(), R)[:, None, :]
    img = torch.zeros(R * R, dtype=torch.float64, device=e.dev)
    img = img.index_add(0, i.reshape(-1), (gy[:, :, None] * gx[:, None, :]).reshape(-1)).reshape(R, R)
    return ((img - e.put(target)) ** 2).mean()


def exact(case, seed):
    """run()'s outputs for a new state in 64 bits.  None for the wrapped
    positions: a bead on the periodic edge may come out on either side."""
    kind = case["kind"]
    if kind in ("step", "grad"):
        e = _Exact([_one(case, seed)])
        cost = case["steps"] * (e.H * e.W / 2.0e6 + e.X.shape[0] / 1.0e6 + 0.15 * (1 + case["mdf"])) * 0.03
        if (cost if kind == "step" else 3 * cost) > 20:
            return None
    if kind == "step":
        with torch.no_grad():
            for _ in range(case["steps"]):
                e.step(case["observe"])
        out = {"x": None, "y": None, "theta": e.th, "disp": e.D}
        if case["fluid"]:
            out["fluid"] = e.f[0] - e.put(np.array(WT))[:, None, None]
        if case["observe"]:
            out["observables"] = e.obs[0]
        return out
    if kind == "grad":
        X0 = e.X
        leaves = [e.th0, e.L0] + [e.put(e.p[k]) for k in ("k_bend", "k_stretch", "k_shear")]
        for v in leaves:
            v.requires_grad_(True)
        e.p.update(zip(("k_bend", "k_stretch", "k_shear"), leaves[2:]))
        for _ in range(case["steps"]):
            e.step()
        e.D.retain_grad()
        target = _target(case, seed)
        loss = _exact_loss(e, case, X0, target)
        loss.backward()
        g = [torch.zeros_like(v) if v.grad is None else v.grad for v in leaves]
        return {"loss": loss.detach().reshape(1), "gx": e.D.grad[:, 0], "gy": e.D.grad[:, 1], "theta0": g[0],
                "L_rest": g[1], "k": torch.stack(g[2:])}
    specs = _specs(case, seed)
    order, groups = list(range(len(specs))), {}
    for k in order:
        groups.setdefault((specs[k].H, specs[k].W), []).append(k)
    if len(groups) * case["steps"] * (0.02 + 0.002 * case["worlds"] / 16) > 20:
        return None
    th, D, obs = [None] * len(specs), [None] * len(specs), [None] * len(specs)
    with torch.no_grad():
        for ks in groups.values():
            e = _Exact([specs[k] for k in ks])
            for _ in range(case["steps"]):
                e.step(case["observe"])
            for m, k in enumerate(ks):
                th[k], D[k], obs[k] = e.th[e.ew == m], e.D[e.w == m], e.obs[m]
    if kind == "batch":
        return {"x": None, "y": None, "theta": torch.cat(th), "disp": torch.cat(D)}
    return {"com_disp": torch.stack([d.mean(0) for d in D]), "observables": torch.stack(obs), "status": None}
