"""Performance cases: the runs a user of this package makes, through its public
calls, from the smallest lattice polled every few steps to the 16384 x 16384
one, with plain 64-bit values of their results to compare against.

A case is a dict of plain values.  ``kind`` is
  "run"     one lattice: reset, initial fields, ``steps`` time steps, the fields
            and the crack history read back (a parameter study's inner loop);
  "poll"    one lattice kept running: ``steps`` more time steps, then the
            fields and the crack are read (a program that watches it as it goes);
  "batch"   many lattices kept running together, then their fields read;
  "adjoint" the loss and its gradients of a recorded run.
"""
import math

import numpy as np
import torch

from paper_2206_12412_gb300 import lbm
from paper_2206_12412_gb300 import workloads as W

BYTES = {"f64": 8, "f32": 4, "f32_lf": 4, "f32_bf16": 4, "f32_f16": 4}
U0 = 1e-3


def _run(name, nx, ny, steps, **more):
    c = {"name": name, "kind": "run", "nx": nx, "ny": ny, "steps": steps, "storage": "f32", "lattice": "D2Q5",
         "bc": "macroscopic", "edges": "strip", "crack": "prescribed", "v_rel": 0.5, "two_tips": False}
    c.update(more)
    return c


def listed():
    return [
        # a small strip watched closely: few steps between reads, all launch and read latency
        _run("poll_256x128", 256, 128, 20, kind="poll", crack="stationary"),
        # the plain FP64 verification problem, its 2000 steps
        _run("plain_128_f64", 128, 128, 2000, storage="f64", crack="stationary"),
        # the K-criterion example with two growing tips and the macroscopic rule on every boundary
        _run("centre_512x192", 512, 192, 5050, bc="macroscopic_edges", crack="example", two_tips=True),
        # a ragged body with periodic sides, link-local crack faces and 16-bit rates
        _run("ragged_1001x777_f16", 1001, 777, 1000, storage="f32_f16", bc="bounceback", edges="periodic",
             crack="prescribed", v_rel=0.3),
        # the K-criterion run on 4096 x 2048
        _run("kcrit_4096x2048", 4096, 2048, 512, crack="kcrit"),
        # the nine-velocity lattice at the same size
        _run("d2q9_4096x2048", 4096, 2048, 256, lattice="D2Q9", crack="kcrit"),
        # an inclined centre crack with the macroscopic rule on its faces
        _run("line_2048x1024", 2048, 1024, 512, crack="line", two_tips=True),
        # the large mixed-precision run, BF16 rates
        _run("large_8192_bf16", 8192, 8192, 100, storage="f32_bf16"),
        # the largest lattice, leapfrog FP32
        _run("large_16384_leapfrog", 16384, 16384, 100, storage="f32_lf"),
        # 256 uneven fracture runs advanced together
        {"name": "batch_256", "kind": "batch", "lattices": 256, "problems": 3, "steps": 500, "storage": "f32"},
        # sensor-misfit gradients with every misfit kept, and with square-root checkpoints
        {"name": "adjoint_1024", "kind": "adjoint", "nx": 1024, "ny": 1024, "steps": 2000, "sensors": 64, "every": 0},
        {"name": "adjoint_ckpt_1024", "kind": "adjoint", "nx": 1024, "ny": 1024, "steps": 2000, "sensors": 64, "every": 45},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["run", "poll", "batch", "adjoint"], [7, 1, 2, 2])[0]
    if kind == "poll":
        return _unnamed(_run("", _log(rng, 64, 1024), _log(rng, 64, 512), rng.randint(8, 64), kind="poll",
                             crack="stationary", storage=rng.choice(["f32", "f64"])))
    if kind == "batch":
        return {"kind": "batch", "lattices": _log(rng, 8, 200), "problems": rng.randrange(1 << 20), "steps": _log(rng, 60, 400),
                "storage": rng.choice(["f32", "f32", "f32_lf"])}
    if kind == "adjoint":
        steps = _log(rng, 300, 1900)
        return {"kind": "adjoint", "nx": _log(rng, 128, 1024), "ny": _log(rng, 96, 1000), "steps": steps,
                "sensors": rng.randint(1, 64), "every": rng.choice([0, int(math.sqrt(steps))])}
    # sizes over the whole range; as many steps as a run of that size takes between outputs
    nx, ny = _log(rng, 96, 12000), _log(rng, 64, 9000)
    steps = max(40, min(3000, int(rng.uniform(0.3, 1.0) * 4e9 / (nx * ny))))
    crack = rng.choice(["prescribed", "prescribed", "kcrit", "kcrit", "stationary", "line"])
    lattice = "D2Q5" if crack == "line" else rng.choice(["D2Q5", "D2Q5", "D2Q5", "D2Q9"])
    plain = lattice == "D2Q9" or crack == "line"
    storage = "f32" if plain else rng.choice(["f32", "f32", "f32_lf", "f32_bf16", "f32_f16", "f64"])
    bc = rng.choice(["macroscopic", "macroscopic", "bounceback"] + ([] if plain else ["macroscopic_edges"]))
    edges = "periodic" if bc == "bounceback" and crack != "line" and rng.random() < 0.5 else "strip"
    return _unnamed(_run("", nx, ny, steps, storage=storage, lattice=lattice, bc=bc, edges=edges, crack=crack,
                         v_rel=round(rng.uniform(0.1, 0.7), 3),
                         two_tips=crack == "line" or (crack == "kcrit" and rng.random() < 0.3)))


def _unnamed(case):
    del case["name"]
    return case


# ------------------------------------------------------------------ problems

def _problem(case):
    """The lattice, crack and loads of a "run" or "poll" case."""
    nx, ny = case["nx"], case["ny"]
    if case["crack"] == "example":
        p = W.kcrit_centre_crack(bc_mode=case["bc"])
        if (nx, ny) != (p["nx"], p["ny"]):
            raise ValueError("the example has a size of its own")
        return p
    sides = "periodic" if case["edges"] == "periodic" else "free"
    p = W.base_problem(nx, ny, bc_mode=case["bc"], edges=(sides, sides, "dirichlet", "dirichlet"))
    p["lattice"] = case["lattice"]
    # held at the displaced edges that the initial strain belongs to
    p["loads"] = [{"edge": "top", "kind": "const", "amp": U0}, {"edge": "bottom", "kind": "const", "amp": -U0}]
    K_C = 0.2 * W.strip_reference_K(p["mu"], U0, float(ny))
    if case["crack"] == "line":
        th = math.radians(20.0)
        half = min(nx, ny) / 8.0
        mx, my = nx / 2 + 0.013, ny / 2 + 0.007
        dx, dy = half * math.cos(th), half * math.sin(th)
        return W.with_line_crack(p, mode="kcrit", start=(mx - dx, my - dy), tip=(mx + dx, my + dy), K_C=K_C,
                                 two_tips=case["two_tips"])
    start = 0.375 * nx if case["two_tips"] or sides == "periodic" else 0.0
    tip = 0.625 * nx if case["two_tips"] or sides == "periodic" else nx / 8.0
    return W.with_crack(p, mode=case["crack"], y=float(ny // 2), x_start=start, x_tip=tip, v_rel=case["v_rel"],
                        K_C=K_C, two_tips=case["two_tips"])


def _batch(case):
    """Uneven problems, the same for every seed, held at the displaced edges from the start as the single runs are."""
    probs = W.batch_problems(case["lattices"], seed=case["problems"])
    for p in probs:
        p["loads"] = [dict(ld, kind="const") for ld in p["loads"]]
    return probs


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _fields(case, seed, dtype, u0=U0):
    """Initial (w, wdot): the strain of the held edges (none for the example, which starts at rest) and smooth waves."""
    nx, ny = case["nx"], case["ny"]
    g = _gen(seed)
    x = (torch.arange(nx, device="cuda", dtype=torch.float64) + 0.5) / nx
    y = (torch.arange(ny, device="cuda", dtype=torch.float64) + 0.5) / ny
    strain = 0.0 if case["crack"] == "example" else u0
    out = []
    for amp, base in ((0.05 * u0, strain), (0.002 * u0, 0.0)):
        f = (base * (2.0 * y - 1.0)).to(dtype)[:, None].repeat(1, nx)
        for k in range(1, 5):
            a, px, py = torch.rand(3, generator=g, device="cuda", dtype=torch.float64)
            mode = (amp * (a - 0.5) * torch.sin(math.pi * k * y + py)).to(dtype)
            f.addr_(mode, torch.cos(2 * math.pi * (k * x + px)).to(dtype))
        out.append(f)
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("run", "poll"):
        p = _problem(case)
        lat = lbm.Lattice(p, case["storage"])
        dtype = torch.float64 if case["storage"] == "f64" else torch.float32
        w, wd = _fields(case, seed, dtype)
        if kind == "poll":
            lat.set_fields(w, wd)
        return {"case": case, "lat": lat, "w": w, "wd": wd, "two": bool(p["crack"].get("two_tips"))}
    if kind == "batch":
        probs = _batch(case)
        lats = [lbm.Lattice(p, case["storage"]) for p in probs]
        for k, (p, lat) in enumerate(zip(probs, lats)):
            lat.set_fields(*_fields(p, seed + 1000 * k, torch.float32, p["loads"][0]["amp"]))
        batch = lbm.Batch(lats)
        batch.tune()
        n = sum(p["nx"] * p["ny"] for p in probs)
        return {"case": case, "batch": batch, "lats": lats,
                "w": torch.empty(n, device="cuda"), "wd": torch.empty(n, device="cuda")}
    a = _adjoint_inputs(case, seed)
    lat = lbm.Lattice(a["problem"], "f32")
    tape = lbm.Tape(lat, a["sensors"], case["steps"], checkpoint_every=case["every"])
    return {"case": case, "lat": lat, "tape": tape, **a}


def _adjoint_inputs(case, seed):
    s = int(seed) % (1 << 30)
    a = W.adjoint_problem(case["nx"], case["ny"], case["steps"], case["sensors"], seeds=(s, s + 1, s + 2))
    w, wd = _fields(a["problem"], seed, torch.float32)
    t = 0.3 * U0 * torch.randn((case["steps"], case["sensors"]), generator=_gen(seed + 5), device="cuda",
                               dtype=torch.float64)
    return {"problem": a["problem"], "sensors": a["sensors"], "targets": t, "w": w, "wd": wd,
            "u": torch.from_numpy(np.ascontiguousarray(a["u_ctl"]))}


def run(state):
    case = state["case"]
    kind, steps = case["kind"], case["steps"]
    if kind in ("run", "poll"):
        lat = state["lat"]
        if kind == "run":
            lat.reset()
            lat.set_fields(state["w"], state["wd"])
        lat.step(steps)
        w, wd = lat.fields_device()
        return {"w": w, "wdot": wd, **_history(state, steps)}
    if kind == "batch":
        state["batch"].step(steps)
        at, state_of = 0, []
        for lat in state["lats"]:
            lbm.lbm_fields(lat.h, lbm.A.FIELD["w"], state["w"].data_ptr() + 4 * at, True, lat.dtype_code)
            lbm.lbm_fields(lat.h, lbm.A.FIELD["wdot"], state["wd"].data_ptr() + 4 * at, True, lat.dtype_code)
            at += lat.nx * lat.ny
            state_of.append(lat.crack_state())
        return {"w": state["w"], "wdot": state["wd"], "K": np.array([s["K"] for s in state_of]),
                "tip_q": np.array([s["tip_q"] for s in state_of])}
    u = state["u"].clone().requires_grad_(True)
    w = state["w"].clone().requires_grad_(True)
    wd = state["wd"].clone().requires_grad_(True)
    loss = lbm.sensor_misfit(state["tape"], "top", u, w, wd, state["targets"])
    loss.backward()
    return {"loss": loss.detach(), "du": u.grad, "dw": w.grad, "dwdot": wd.grad}


def _history(state, steps):
    h = state["lat"].history(steps)
    out = {"K": h["K"], "tip_q": h["tip_q"], "npairs": h["npairs"]}
    if state["two"]:
        hl = state["lat"].history_left(steps)
        out.update(K_left=hl["K"], tip_q_left=hl["tip_q"])
    return out


def work(case):
    """The initial fields read and the final ones written once; per site and step the update's sums and products
    (eight with four neighbours, fourteen with eight)."""
    kind, steps = case["kind"], case["steps"]
    if kind == "batch":
        sites = 320 * 640 * case["lattices"]   # the mean of the sizes that are drawn
    else:
        sites = case["nx"] * case["ny"]
    planes = 4 * BYTES[case.get("storage", "f32")] * sites
    flops = float(sites) * steps * (14 if case.get("lattice") == "D2Q9" else 8)
    if kind == "adjoint":
        return {"bytes": planes + 8 * steps * (2 + case["sensors"]), "flops": 2 * flops}
    return {"bytes": planes + 28 * steps, "flops": flops}


# ------------------------------------------- the same results in plain 64 bits

def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        if case["lattices"] * case["steps"] > 20000:
            return None
        outs = []
        for k, p in enumerate(_batch(case)):
            w, wd = _fields(p, seed + 1000 * k, torch.float32, p["loads"][0]["amp"])
            outs.append(_march(p, w.double(), wd.double(), case["steps"]))
        return {"w": torch.cat([o["w"].reshape(-1) for o in outs]), "wdot": torch.cat([o["wdot"].reshape(-1) for o in outs]),
                "K": np.array([o["K"][-1] for o in outs]), "tip_q": None}
    if kind == "adjoint":
        return _exact_adjoint(case, seed)
    if case["crack"] == "line":
        return None
    p = _problem(case)
    dtype = torch.float64 if case["storage"] == "f64" else torch.float32
    w, wd = (f.double() for f in _fields(case, seed, dtype))
    o = _march(p, w, wd, case["steps"])
    out = {"w": o["w"], "wdot": o["wdot"], "K": o["K"], "tip_q": None, "npairs": None}
    if p["crack"].get("two_tips"):
        out.update(K_left=o["K_left"], tip_q_left=None)
    return out


def _load(p, edge, n):
    """w* of an edge at t_n (0 where none is given)."""
    for ld in p["loads"]:
        if ld["edge"] == edge:
            if ld["kind"] == "const":
                return ld["amp"]
            if ld["kind"] == "series":
                return ld["series"][min(n, len(ld["series"]) - 1)]
            if ld["kind"] == "halfsine":
                return 0.0 if n >= ld["t"] else ld["amp"] * math.sin(math.pi * n / ld["t"])
    return 0.0


class _Tip:
    """One growing end: the tip on a 2^-32 grid, its speed and its records."""

    def __init__(self, x, sign):
        self.q, self.sign, self.v, self.stopped, self.K = round(x * 2 ** 32), sign, 0.0, False, []


def _crack_step(p, tips, cut, nx, opening):
    """K from the opening behind each end, the criterion and the advance, on the columns cut = [first, last]."""
    c = p["crack"]
    cs = math.sqrt(p["mu"] / p["rho"])
    half = 1 << 31
    for t in tips:
        r_min = c["r0"] / (1.0 - t.v)
        x = t.q / 2 ** 32
        num = den = 0.0
        for i in range(int(x) - 64, int(x) + 65) if r_min < 60 else ():
            r = t.sign * (x - (i + 0.5))
            if cut[0] <= i <= cut[1] and r_min <= r < r_min + c["fit_width"]:
                s = math.sqrt(r / (2.0 * math.pi))
                num += opening[i] * s
                den += s * s
        K = p["mu"] / 4.0 * num / den if den else 0.0
        t.K.append(K)
        grow = c["mode"] == "prescribed" or (c["mode"] == "kcrit" and den > 0 and abs(K) > c["K_C"])
        v = 0.0
        if grow:
            v = c["v_rel"] if c["mode"] == "prescribed" else c["v_max"] * math.tanh(math.sqrt((abs(K) / c["K_C"]) ** 4 - 1.0))
        if t.stopped:
            grow, v = False, 0.0
        t.v = c["v_rel"] if c["mode"] == "prescribed" else v
        if grow:
            q = t.q + t.sign * round(v * cs * 2 ** 32)
            if t.sign > 0:
                if q >= nx << 32:
                    q, t.stopped = nx << 32, True
                cut[1] = max(cut[1], min((q - half) >> 32, nx - 1))
            else:
                if q <= 0:
                    q, t.stopped = 0, True
                cut[0] = min(cut[0], max((q - half + (1 << 32) - 1) >> 32, 0))
            t.q = q


def _shifted(p, w, dx, dy, ws):
    """The value each site receives over the link to (i + dx, j + dy): the neighbour's, the site's own (bounce-back)
    where the link leaves through a free edge, 2 w* - w where through a Dirichlet edge; periodic sides wrap."""
    e = p["edges"]
    ny, nx = w.shape
    nb = torch.roll(w, (-dy, -dx), (0, 1))
    lr, bt = e[0] if dx < 0 else e[1], e[2] if dy < 0 else e[3]
    if dy:
        j = 0 if dy < 0 else ny - 1
        nb[j] = 2.0 * ws[2 if dy < 0 else 3] - w[j] if bt == "dirichlet" else w[j]
    if dx and lr != "periodic":
        i = 0 if dx < 0 else nx - 1
        inner = slice(None) if not dy else (slice(1, None) if dy < 0 else slice(None, -1))
        nb[inner, i] = w[inner, i]
    return nb


def _march(p, w, wd, steps):
    """`steps` time steps of a body with a crack along +x from (w, wdot), by the equations of the method."""
    nx, ny, c = p["nx"], p["ny"], p["crack"]
    g = p["mu"] / p["rho"]
    jc = int(c["y"])
    nine = p.get("lattice") == "D2Q9"
    start_q = round(c["x_start"] * 2 ** 32)
    tips = [_Tip(c["x_tip"], +1)] + ([_Tip(c["x_start"], -1)] if c["two_tips"] else [])
    cut = [max((start_q - (1 << 31) + (1 << 32) - 1) >> 32, 0), min((tips[0].q - (1 << 31)) >> 32, nx - 1)]
    for t in tips:
        t.v = c["v_rel"] if c["mode"] == "prescribed" else 0.0
    macro = p["bc_mode"] != "bounceback"
    for n in range(steps):
        ws = [_load(p, e, n) for e in ("left", "right", "bottom", "top")]
        lq = tips[1].q if c["two_tips"] else start_q
        f, l = cut
        # diagonal links (nine velocities) cross the crack line at x = m, severed for lq <= m <= tip
        m0, m1 = max(-(-lq >> 32), 1), min(tips[0].q >> 32, nx - 1)
        acc = torch.zeros_like(w)
        links = [(1, 0), (-1, 0), (0, 1), (0, -1)] + ([(1, 1), (-1, 1), (1, -1), (-1, -1)] if nine else [])
        for dx, dy in links:
            nb = _shifted(p, w, dx, dy, ws)
            if dy:
                j = jc - 1 if dy > 0 else jc
                if not dx:
                    nb[j, f:l + 1] = w[j, f:l + 1]
                elif m1 >= m0:
                    s = slice(m0 - 1, m1) if dx > 0 else slice(m0, m1 + 1)
                    nb[j, s] = w[j, s]
            nb.sub_(w)
            acc.add_(nb, alpha=(1.0 / 6.0 if dx and dy else 2.0 / 3.0) if nine else 1.0)
        wd = wd + g * acc
        new = w + wd
        if macro:
            face = [(f, l + 1)]
            if nine and m1 >= m0:
                face.append((m0 - 1, m1 + 1))
            old = new.clone()
            for a, b in face:
                for j, s in ((jc - 1, -1), (jc, 1)):
                    if b > a:
                        new[j, a:b] = 1.5 * old[j + s, a:b] - 0.5 * old[j + 2 * s, a:b]
            rows = slice(jc - 1, jc + 1)
            wd[rows] = new[rows] - w[rows]
        if p["bc_mode"] == "macroscopic_edges":
            _edge_rule(p, w, new, wd, n, cut, jc)
        w = new
        openings = (w[jc] - w[jc - 1]).cpu().numpy() if nx <= 1024 else None
        if openings is None:
            openings = _Window(w, jc, tips, nx)
        _crack_step(p, tips, cut, nx, openings)
    return {"w": w, "wdot": wd, "K": np.array(tips[0].K), "K_left": np.array(tips[-1].K)}


class _Window:
    """The openings of the columns near each tip, by column."""

    def __init__(self, w, jc, tips, nx):
        self.parts = []
        for t in tips:
            a, b = max((t.q >> 32) - 64, 0), min((t.q >> 32) + 66, nx)
            self.parts.append((a, (w[jc, a:b] - w[jc - 1, a:b]).cpu().numpy()))

    def __getitem__(self, i):
        for a, part in self.parts:
            if a <= i < a + len(part):
                return part[i - a]
        raise IndexError(i)


def _edge_rule(p, w, new, wd, n, cut, jc):
    """The macroscopic rule on the outer edges: the quadratic along the inward normal at each edge site."""
    ny, nx = w.shape
    old = new.clone()
    ws = [_load(p, e, n + 1) for e in ("left", "right", "bottom", "top")]
    kind = p["edges"]

    def rule(e, a, b):
        if kind[e] == "dirichlet":
            return 8.0 / 15.0 * ws[e] + 2.0 / 3.0 * a - 0.2 * b
        return 1.5 * a - 0.5 * b

    left, right = rule(0, old[:, 1], old[:, 2]), rule(1, old[:, -2], old[:, -3])
    bottom, top = rule(2, old[1], old[2]), rule(3, old[-2], old[-3])
    new[0, 1:-1], new[-1, 1:-1] = bottom[1:-1], top[1:-1]
    new[1:-1, 0], new[1:-1, -1] = left[1:-1], right[1:-1]
    for i, col in ((0, left), (nx - 1, right)):
        if cut[0] <= i <= cut[1]:
            new[jc, i] = 1.5 * col[jc + 1] - 0.5 * col[jc + 2]
            new[jc - 1, i] = 1.5 * col[jc - 2] - 0.5 * col[jc - 3]
        for j, row, e, s in ((0, bottom, 2, 1), (ny - 1, top, 3, -1)):
            h = 0 if i == 0 else 1
            if kind[h] == "dirichlet" and kind[e] != "dirichlet":
                d = 1 if i == 0 else -1
                new[j, i] = rule(h, row[i + d], row[i + 2 * d])
            else:
                new[j, i] = rule(e, col[j + s], col[j + 2 * s])
    for s in ((0, slice(None)), (-1, slice(None)), (slice(None), 0), (slice(None), -1)):
        wd[s] = new[s] - w[s]


def _exact_adjoint(case, seed):
    """Loss and gradients by reverse accumulation through the same steps in 64 bits (the schedule is prescribed)."""
    if case["nx"] * case["ny"] * case["steps"] > 3e9:
        return None
    a = _adjoint_inputs(case, seed)
    p, c = a["problem"], a["problem"]["crack"]
    g = p["mu"] / p["rho"]
    nx, jc, steps = p["nx"], int(c["y"]), case["steps"]
    u = a["u"].double().cuda()
    si, sj = (torch.from_numpy(np.ascontiguousarray(a["sensors"][:, k])).long().cuda() for k in (0, 1))
    tip = _Tip(c["x_tip"], +1)
    cut = [0, min((tip.q - (1 << 31)) >> 32, nx - 1)]
    cuts, w, wd = [], a["w"].double(), a["wd"].double()
    res = []
    for n in range(steps):   # forward
        l = cut[1]
        cuts.append(l)
        acc = _strip_laplacian(w, jc, l)
        acc[0] -= 2.0 * w[0]
        acc[-1] += 2.0 * (u[n] - w[-1])
        wd = wd + g * acc
        new = w + wd
        for j, s in ((jc - 1, -1), (jc, 1)):
            new[j, :l + 1] = 1.5 * new[j + s, :l + 1] - 0.5 * new[j + 2 * s, :l + 1]
            wd[j] = new[j] - w[j]
        w = new
        res.append(w[sj, si] - a["targets"][n])
        _crack_step(p, [tip], cut, nx, _Zero())
    loss = torch.stack(res).square().sum()
    gw, gd = torch.zeros_like(w), torch.zeros_like(w)   # d loss / d (w, wdot) after step n
    du = torch.zeros(steps, dtype=torch.float64, device="cuda")
    for n in reversed(range(steps)):
        l = cuts[n]
        gw.index_put_((sj, si), 2.0 * res[n], accumulate=True)
        back = torch.zeros(2, nx, dtype=torch.float64, device="cuda")   # wdot_B = w_B - w(t): straight to the old w
        for k, (j, s) in enumerate(((jc - 1, -1), (jc, 1))):
            t = gw[j, :l + 1] + gd[j, :l + 1]
            back[k, :l + 1] = -gd[j, :l + 1]
            gw[j + s, :l + 1] += 1.5 * t
            gw[j + 2 * s, :l + 1] -= 0.5 * t
            gw[j, :l + 1] = 0.0
            gd[j, :l + 1] = 0.0
        gd = gd + gw
        du[n] = 2.0 * g * gd[-1].sum()
        acc = _strip_laplacian(gd, jc, l)   # the sum over links is its own transpose
        acc[0] -= 2.0 * gd[0]
        acc[-1] -= 2.0 * gd[-1]
        gw = gw + g * acc
        gw[jc - 1:jc + 1] += back
    return {"loss": loss, "du": du.cpu(), "dw": gw, "dwdot": gd}


class _Zero:
    def __getitem__(self, i):
        return 0.0


def _strip_laplacian(w, jc, last):
    """Sum over intact links of (neighbour - own); columns 0..last of the links between rows jc - 1 and jc are severed."""
    acc = torch.zeros_like(w)
    d = w[:, 1:] - w[:, :-1]
    acc[:, :-1] += d
    acc[:, 1:] -= d
    d = w[1:] - w[:-1]
    d[jc - 1, :last + 1] = 0.0
    acc[:-1] += d
    acc[1:] -= d
    return acc
