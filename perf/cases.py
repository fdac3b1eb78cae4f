"""What a user of this library has it do, as cases that can be timed.

A case is a dict of plain values. ``prepare`` makes what a program holds before
the call (the simulations, their batch, the buffers that results go to),
``run`` is one pass through the public entry points, and ``exact`` is what that
pass returns as plain torch arithmetic in 64 bits gives it.

Kinds of pass:

* ``single``: one resident lattice is advanced by ``steps`` steps; then either
  the front is read back with a wait (``read = "front"``, the loop that samples
  the roughness), or the front goes to pinned memory and the density and
  velocity fields to device arrays (``read = "fields"``);
* ``batch``: many resident lattices are advanced together, then each member's
  front (and with ``read = "fields"`` its fields) is read;
* ``whole``: a run from its parameters to its results: the lattice is created,
  stepped with the front recorded at every step, its fields taken, and closed.

Advancing rear walls keep the active window about as tall after many passes as
in the first one, so a pass costs the same whenever it is run.
"""
from __future__ import annotations

import math

import torch

from paper_2303_02210_gb300 import workloads as wl
from paper_2303_02210_gb300.lbm import Batch, Simulation

ELEM = {"fp32": 4, "fp64": 8, "fp16": 2, "bf16": 2}


def listed():
    return [
        # the smallest call: one step of the 128-column lattice, then its front on the host; latency is all there is
        dict(name="small_128_fp32", kind="single", width=128, height=512, front_row=52, steps=1, read="front"),
        # the roughness runs' lattice, 1024 columns of bulk growth, sampled every ten steps
        dict(name="kpz_1024_fp32", kind="single", width=1024, height=1024, front_row=64, steps=10, read="fields"),
        # the benchmark's lattice: 4096 columns by about a thousand active rows, growth within 8 rows of the front
        dict(name="edge_4096_fp32", kind="single", width=4096, height=2048, front_row=1024, growth="edge", gap=1000.0,
             front="sinusoidal", steps=20, read="fields"),
        # twice as wide: the largest single lattice
        dict(name="edge_8192_fp32", kind="single", width=8192, height=2048, front_row=1024, growth="edge", gap=1000.0,
             front="sinusoidal", steps=20, read="fields"),
        # the same with FP16 population storage
        dict(name="edge_8192_fp16", kind="single", width=8192, height=2048, front_row=1024, growth="edge", gap=1000.0,
             front="sinusoidal", precision="fp16", steps=20, read="fields"),
        # density-dependent growth (the unstable fronts) on an odd size, BF16 storage
        dict(name="density_1501_bf16", kind="single", width=1501, height=777, front_row=190, growth="density",
             precision="bf16", steps=10, read="fields"),
        # the benchmark's lattice on the paper's triangular D2Q7
        dict(name="edge_4096_d2q7", kind="single", lattice="d2q7", width=4096, height=2048, front_row=1024,
             growth="edge", gap=1000.0, front="sinusoidal", steps=20, read="fields"),
        # the FP64 path, the paper's own parameter list with its heavy noise
        dict(name="paper_512_fp64", kind="single", width=512, height=1024, front_row=64, scale="paper", rate=1e-4, negfix="rescale",
             precision="fp64", steps=10, read="fields"),
        # 256 uneven realisations (widths 256..2048) together, as the roughness statistics need them
        dict(name="ensemble_256_fp32", kind="batch", members="ensemble", n=256, steps=40, read="fields"),
        # a full slot batch of the serving loop: widths 128..4096, three growth modes, FP16 storage
        dict(name="serving_256_fp16", kind="batch", members="serving", n=256, precision="fp16", steps=40, read="front"),
        # the KPZ check: 32 seeds of each width 64..512 on D2Q7 in the paper's regime, sampled every ten steps
        dict(name="kpz_128_d2q7", kind="batch", members="kpz", n=128, lattice="d2q7", steps=10, read="front"),
        # a whole short run from parameters to results, the front recorded at every step
        dict(name="whole_2048_fp32", kind="whole", width=2048, height=1024, front_row=512, growth="edge", gap=500.0,
             front="sinusoidal", steps=50, read="fields"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["single"] * 6 + ["batch"] * 3 + ["whole"])
    if kind == "batch":
        members = rng.choice(["ensemble", "serving", "kpz"])
        n = int(_log(rng, 2, 256))
        c = dict(kind="batch", members=members, n=n, steps=rng.randint(5, 40), read=rng.choice(["front", "fields"]))
        if members == "kpz":
            c.update(lattice="d2q7", read="front")
        else:
            c.update(precision=rng.choice(["fp32", "fp32", "fp16", "bf16"]), salt=rng.randint(0, 999))
        return c
    W = int(_log(rng, 33, 8192))
    if rng.random() < 0.5:
        W = max(64, W // 32 * 32)
    growth = rng.choice(["bulk", "edge", "density", "band"])
    thin = rng.random() < 0.5
    rows = rng.randint(60, 120) if thin else int(_log(rng, 120, 1024))
    lattice = rng.choice(["d2q9", "d2q9", "d2q9", "d2q7"])
    precision = rng.choice(["fp32", "fp32", "fp64"] if lattice == "d2q7" else ["fp32", "fp32", "fp32", "fp16", "bf16", "fp64"])
    if precision == "fp64":
        W, rows = min(W, 2048), min(rows, 300)
    c = dict(kind=kind, width=W, height=rows + rng.randint(500, 1000), front_row=rows, growth=growth, lattice=lattice,
             precision=precision, gap=float(max(50, rows - 12)), rate=_log(rng, 1e-5, 1e-4), steps=rng.randint(1, 20),
             read=rng.choice(["front", "fields"]) if kind == "single" else "fields",
             front=rng.choice(["flat", "sinusoidal"]), negfix=rng.choice(["literal", "literal", "rescale"]),
             sigma=rng.choice([0.01, 0.01, 0.01, 0.0]))
    return c


# ---------------------------------------------------------------- parameters
def _params(c, seed):
    """The parameter dictionary of a one-lattice case."""
    base = wl.paper_params if c.get("scale") == "paper" else wl.base_params
    return base(width=c["width"], height=c["height"], tau=1.0 if c.get("scale") == "paper" else 0.8,
                growth_rate=c.get("rate", 1e-4), growth_mode=c.get("growth", "bulk"), edge_depth=8,
                front_kind=c.get("front", "flat"), front_row=float(c["front_row"]),
                front_amp=1.0 if c.get("front") == "sinusoidal" else 0.5, wall_mode="advance",
                wall_min_gap=float(c.get("gap", 50.0)), negfix_mode=c.get("negfix", "literal"),
                sigma=c.get("sigma", 0.01), lattice=c.get("lattice", "d2q9"), seed=seed, sim_id=seed % 997)


def _members(c, seed):
    """The members' parameter dictionaries: the shapes are the case's own, the random streams the seed's."""
    n, salt = c["n"], c.get("salt", 1)
    if c["members"] == "ensemble":
        ps = wl.ensemble(n, seed=salt)
    elif c["members"] == "serving":
        ps = [p for _, p, _, _ in wl.serving_trace(n, seed=salt)]
    else:
        ps = [wl.paper_params(width=(64, 128, 256, 512)[i % 4], height=4096, lattice="d2q7", growth_mode="bulk",
                              wall_mode="advance", front_row=60.0, front_amp=0.5, negfix_mode="rescale")
              for i in range(n)]
    return [dict(p, seed=seed * 1000 + i, sim_id=i) for i, p in enumerate(ps)]


# ---------------------------------------------------------------- the pass
def _front_buffers(widths):
    return (torch.empty(sum(widths), dtype=torch.int32, pin_memory=True),
            torch.empty(len(widths), 2, dtype=torch.int64, pin_memory=True))


def _field_buffers(nodes):
    return [torch.empty(nodes, dtype=torch.float64, device="cuda") for _ in range(3)]


def prepare(case, seed):
    c, precision = case, case.get("precision", "fp32")
    st = {"case": c, "seed": seed}
    if c["kind"] == "batch":
        ps = _members(c, seed)
        sims = [Simulation(p, precision=precision) for p in ps]
        if c["members"] == "serving":  # the serving loop's slot batch
            batch = Batch.empty(256, precision, "d2q9")
            for s in sims:
                batch.attach(s)
        else:
            batch = Batch(sims)
        st.update(batch=batch, sims=sims)
    else:
        ps = [_params(c, seed)]
        if c["kind"] == "single":
            st.update(sims=[Simulation(ps[0], precision=precision)])
        else:
            st.update(params=ps[0])
    widths = [p["width"] for p in ps] if c["kind"] != "whole" else [ps[0]["width"]] * c["steps"]
    st["h"], st["sums"] = _front_buffers(widths)
    st["hs"], st["ss"] = list(torch.split(st["h"], widths)), list(st["sums"])
    if c["read"] == "fields":
        nodes = [p["width"] * p["height"] for p in ps]
        st["fields"] = _field_buffers(sum(nodes))
        st["views"] = list(zip(*[torch.split(f, nodes) for f in st["fields"]]))
    return st


def run(state):
    st, c = state, state["case"]
    if c["kind"] == "whole":
        with Simulation(st["params"], precision=c.get("precision", "fp32")) as sim:
            for h, s in zip(st["hs"], st["ss"]):
                sim.step(1)
                sim.lbm_front_heights_async(h, s)
            sim.lbm_fields_device(*st["views"][0])
            sim.sync()
        return {"h": st["h"], "sums": st["sums"], "rho": st["fields"][0], "ux": st["fields"][1], "uy": st["fields"][2]}
    if c["kind"] == "single" and c["read"] == "front":
        sim = st["sims"][0]
        sim.step(c["steps"])
        h, hbar, w = sim.front_heights()
        return {"h": h, "hbar": hbar, "w": w}
    if c["kind"] == "single":
        st["sims"][0].step(c["steps"])
    else:
        st["batch"].step(c["steps"])
    for sim, h, s in zip(st["sims"], st["hs"], st["ss"]):
        sim.lbm_front_heights_async(h, s)
    out = {"h": st["h"], "sums": st["sums"]}
    if c["read"] == "fields":
        for sim, v in zip(st["sims"], st["views"]):
            sim.lbm_fields_device(*v)
        out.update(rho=st["fields"][0], ux=st["fields"][1], uy=st["fields"][2])
    return out


def work(case):
    """Every population of the active window read and written once a step (the window: from the rear wall to two rows
    above the front), the fields read from the populations and written once, the fronts written once."""
    c, precision = case, case.get("precision", "fp32")
    ps = _members(c, 1) if c["kind"] == "batch" else [_params(c, 1)]
    by = fl = 0
    for p in ps:
        q = 7 if p["lattice"] == "d2q7" else 9
        wall = max(0, int(p["front_row"] - p["wall_min_gap"])) if p["wall_mode"] == "advance" else 0
        active = p["width"] * (min(p["height"], int(p["front_row"]) + 3) - wall)
        by += c["steps"] * active * 2 * q * ELEM[precision] + 4 * p["width"]
        fl += c["steps"] * active * 25 * q
        if c["read"] == "fields":
            by += p["width"] * p["height"] * (q * ELEM[precision] + 24)
        if c["kind"] == "whole":
            by += 2 * p["width"] * p["height"] * q * ELEM[precision] + 4 * p["width"] * (c["steps"] - 1)
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------- the same in 64 bits
M32 = 0xFFFFFFFF


def _philox(n, a, stream, sim, seed):
    """Philox4x32-10 on the counters (n, a, stream, sim), n an int64 tensor."""
    def mul(x, m):
        lo = (x * m) & M32
        hi = (((x * (m >> 16)) + ((x * (m & 0xFFFF)) >> 16)) >> 16) & M32
        return hi, lo
    c0, c1 = n & M32, torch.full_like(n, a & M32)
    c2, c3 = torch.full_like(n, stream), torch.full_like(n, sim & M32)
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        h0, l0 = mul(c0, 0xD2511F53)
        h1, l1 = mul(c2, 0xCD9E8D57)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c0, c1, c2, c3


def _u01(v):
    return (v.double() + 0.5) * 2.0 ** -32


class _Exact:
    """One lattice in 64-bit torch arithmetic, walls in y."""

    def __init__(self, p):
        self.p, self.t = p, 0
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        W, H = self.W, self.H = p["width"], p["height"]
        self.d7 = p["lattice"] == "d2q7"
        s = math.sqrt(3) / 2
        if self.d7:
            self.e = [(0, 0), (1, 0), (.5, s), (-.5, s), (-1, 0), (-.5, -s), (.5, -s)]
            self.opp, self.w = [0, 4, 5, 6, 1, 2, 3], [.5] + [1 / 12] * 6
            self.pairs, self.coef, self.bits = [(1, 4), (2, 5), (3, 6)], (4, 8, 2), 18
        else:
            self.e = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
            self.opp, self.w = [0, 3, 4, 1, 2, 7, 8, 5, 6], [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
            self.pairs, self.coef, self.bits = [(1, 3), (2, 4), (5, 7), (6, 8)], (3, 4.5, 1.5), 14
        self.Q = len(self.e)
        x = torch.arange(W, device=dev)
        if p["front_kind"] == "flat":
            h0 = p["front_row"] + p["front_amp"] * (2 * _u01(_philox(x, 0, 2, p["sim_id"], p["seed"])[0]) - 1)
        else:
            k = torch.arange(p["front_kmin"], p["front_kmax"] + 1, device=dev)
            phi = 2 * math.pi * _u01(_philox(k, 1, 2, p["sim_id"], p["seed"])[0])
            S = torch.sin(2 * math.pi * k.double()[:, None] * x.double() / W + phi[:, None]).sum(0)
            h0 = p["front_row"] + p["front_amp"] * S / S.abs().max()
        rows = torch.ceil(h0).clamp(0, H)
        self.y = torch.arange(H, device=dev)[:, None].expand(H, W)
        self.n = self.y * W + x
        rho = torch.full((H, W), float(p["rho_init"]), dtype=torch.float64, device=dev)
        if p["rho_jitter"]:
            rho = rho * (1 + p["rho_jitter"] * (2 * _u01(_philox(self.n, 2, 2, p["sim_id"], p["seed"])[0]) - 1))
        rho = torch.where(self.y < rows, rho, 0.0)
        self.f = torch.stack([w * rho for w in self.w])
        self.mask, self.y_r, self.carry = rho >= p["rho_c"], 0, 0.0
        self.observe()

    def fix(self, a):
        return int(torch.round(a * 2.0 ** 24).to(torch.int64).sum())

    def observe(self):
        p = self.p
        self.h = torch.where(self.mask, self.y + 1, 0).amax(0)
        S1, S2 = int(self.h.sum()), int((self.h * self.h).sum())
        self.sums, self.hbar = (S1, S2), S1 / self.W
        self.width = math.sqrt(self.W * S2 - S1 * S1) / self.W
        if p["wall_mode"] == "advance":
            gap = max(p["wall_min_gap"], p["wall_w_factor"] * self.width)
            self.y_r = max(self.y_r, int(min(math.floor(self.hbar - gap), self.H - 1)))
        self.mass = self.fix(self.f.sum(0)[self.y_r:]) * 2.0 ** -24

    def stream(self):
        """Pull streaming; across a wall a node gets its own opposite population."""
        f, out = self.f, []
        odd = (self.y & 1).bool()
        for q in range(self.Q):
            if self.d7 and q not in (0, 1, 4):
                up = q in (2, 3)
                g = torch.roll(f[q], 1 if up else -1, 0)
                even_dx, odd_dx = (-1, 0) if q in (2, 6) else (0, 1)
                g = torch.where(odd, torch.roll(g, -odd_dx, 1), torch.roll(g, -even_dx, 1))
                ey = 1 if up else -1
            else:
                ex, ey = (int(v) for v in self.e[q])
                g = torch.roll(f[q], (ey, ex), (0, 1))
            own = self.y == self.y_r if ey == 1 else (self.y == self.H - 1 if ey == -1 else None)
            out.append(g if own is None else torch.where(own, f[self.opp[q]], g))
        return torch.stack(out)

    def divide(self, fs):
        p, W = self.p, self.W
        if p["growth_mode"] == "none":
            return
        x_ns = p["growth_rate"] * self.mass / p["rho_cell"] + self.carry
        ns = math.floor(x_ns)
        self.carry = x_ns - ns
        lo, hi = self.y_r, int(self.h.max())
        if p["growth_mode"] == "edge":
            lo = max(lo, int(self.h.min()) - p["edge_depth"])
        elif p["growth_mode"] == "band":
            hi = min(hi, self.y_r + p["band_rows"])
        win = max(0, hi - lo) * W
        if ns <= 0 or win <= 0:
            return
        rho = fs.sum(0).reshape(-1)
        k = torch.arange(64 * ns + 1024, device=rho.device)
        r = _philox(k, self.t, 1, p["sim_id"], p["seed"])
        node = lo * W + ((r[0] * win) >> 32)
        pair = (r[1] * len(self.pairs)) >> 32
        rs = rho[node]
        if p["growth_mode"] == "density":
            ok = (rs > p["rho_c"]) & (_u01(r[2]) < 1 - rs / p["rho0"])
        else:
            ok = rs >= p["rho_c"]
            if p["growth_mode"] == "edge":
                ok &= self.h[node % W] - node // W <= p["edge_depth"]
        at = torch.nonzero(ok)[:ns, 0]
        flat = fs.reshape(self.Q, -1)
        for i, ab in enumerate(self.pairs):
            sel = node[at[pair[at] == i]]
            add = torch.bincount(sel, minlength=flat.shape[1]).double() * (p["rho_cell"] / 2)
            for q in ab:
                flat[q] += add

    def step(self):
        p, Q = self.p, self.Q
        fs = self.stream()
        self.divide(fs)
        rho = fs.sum(0)
        occ = rho >= p["rho_c"]
        safe = torch.where(occ, rho, 1.0)
        e = torch.tensor(self.e, dtype=torch.float64, device=fs.device)
        us = [(1 - p["mu"]) * sum(e[q, a] * fs[q] for q in range(Q)) / safe for a in (0, 1)]
        uu, (c1, c2, c3) = us[0] ** 2 + us[1] ** 2, self.coef
        fo = torch.empty_like(fs)
        for q in range(Q):
            eu = e[q, 0] * us[0] + e[q, 1] * us[1]
            fo[q] = fs[q] - (fs[q] - self.w[q] * rho * (1 + c1 * eu + c2 * eu * eu - c3 * uu)) / p["tau"]
        if p["sigma"]:
            words = _philox(self.n, self.t, 16, p["sim_id"], p["seed"])
            us = []
            for q in range(Q):
                j, o = divmod(self.bits * q, 32)
                two = words[j] | ((words[j + 1] & 0x7FFFFFFF) << 32 if j < 3 else 0)
                us.append((((two >> o) & ((1 << self.bits) - 1)).double() + 0.5) * 2.0 ** -self.bits)
            mean = sum(us) / Q
            for q in range(Q):
                fo[q] += 2 * p["sigma"] * (us[q] - mean)
        if p["negfix_mode"] == "literal":
            bad = fo[0] < 0
            r0 = fo.sum(0)
            fo[0] = torch.where(bad, 0.0, fo[0])
            scale = torch.where(bad, r0 / torch.where(bad, fo.sum(0), 1.0), 1.0)
            fo *= scale
            for q in range(1, Q):
                a = (-fo[q]).clamp(min=0)
                fo[self.opp[q]] += a
                fo[q] += a
        else:
            r0, neg = fo.sum(0), (fo < 0).any(0)
            cut = fo.clamp(min=0)
            fo = torch.where(neg, cut * (r0 / torch.where(neg, cut.sum(0), 1.0)), fo)
        fo = torch.where(occ, fo, fs[self.opp])
        fo[:, :self.y_r] = self.f[:, :self.y_r]
        occ[:self.y_r] = self.mask[:self.y_r]
        self.f, self.mask, self.t = fo, occ, self.t + 1
        self.observe()

    def fields(self):
        rho = self.f.sum(0)
        e = torch.tensor(self.e, dtype=torch.float64, device=rho.device)
        safe = torch.where(rho != 0, rho, 1.0)
        return [rho] + [sum(e[q, a] * self.f[q] for q in range(self.Q)) / safe for a in (0, 1)]


def exact(case, seed):
    c = case
    ps = _members(c, seed) if c["kind"] == "batch" else [_params(c, seed)]
    if c["kind"] == "batch" and (c["n"] * c["steps"] > 1500 or c["read"] != "fields"):
        return None  # too long, or whole numbers alone
    fields = []
    for p in ps:
        s = _Exact(p)
        for _ in range(c["steps"]):
            s.step()
        if c["kind"] == "single" and c["read"] == "front":
            return {"h": None, "hbar": s.hbar, "w": s.width}
        fields.append([v.reshape(-1) for v in s.fields()])
    rho, ux, uy = (torch.cat(v) for v in zip(*fields))
    return {"h": None, "sums": None, "rho": rho, "ux": ux, "uy": uy}
