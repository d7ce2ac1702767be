"""The work a user of this library has it do, as cases that can be timed and compared.

Every case goes through the public Python API (Hierarchy, Batch, Field).  Inputs are
made from a seed with plain torch on the GPU: Gaussian fields with P(k) ~ k^-2 on the
periodic base, and on every nest the parent's field interpolated plus fresh small-scale
noise, at the amplitudes initial conditions have (a few per cent).
"""

import math

import numpy as np
import torch

import paper_1103_6031_gb300 as mg

BOX = 100.0  # Mpc/h, the box of the library's own workloads
ROOM = 10_500_000  # level-cells of the largest case (128^3 base + 4 nests of 128^3)


# ---- cases ---------------------------------------------------------------------------


def listed():
    def case(name, kind, base, nests="", order=6, precision="fp64", tol=3e-8, inner=4, host=False,
             members=0):
        return {"name": name, "kind": kind, "base": base, "nests": nests, "order": order,
                "precision": precision, "tol": tol, "inner": inner, "host": host,
                "members": members}

    deep = "128x128x128@36,26,34;128x128x128@37,22,29;128x128x128@22,44,31;128x128x128@40,30,24"
    return [
        # one small periodic solve to the default tolerance: a quick look, a test run; launches
        # and host round trips decide it
        case("solve_unigrid64", "solve", "64x64x64", order=2, tol=1e-10),
        # a small zoom with odd offsets and uneven sides at order 4: a pilot run
        case("step_ragged_o4", "step", "40x48x56", "36x28x44@11,17,13;22x30x26@6,5,9", order=4),
        # a periodic box without refinement, uneven sides: plain (unigrid) initial conditions
        case("step_unigrid", "step", "192x160x224"),
        # base and one nest of the same size: the usual zoom
        case("step_zoom2", "step", "128x128x128", "128x128x128@32,32,32"),
        # the deepest and largest single hierarchy, in both precisions
        case("step_deep", "step", "128x128x128", deep),
        case("step_deep_mixed", "step", "128x128x128", deep, precision="mixed", tol=1e-8, inner=3),
        # one request of a serving mix: inputs and results in pinned host memory
        case("request_mixed", "step", "64x64x64", "56x64x60@14,15,18;48x44x52@12,21,17",
             precision="mixed", tol=1e-8, host=True),
        # many uneven hierarchies at once: an ensemble of zooms
        case("batch_mixed", "batch", "", precision="mixed", tol=1e-8, members=16),
        # the 2LPT source of a given potential, one large periodic level
        case("tau_256", "tau", "256x256x256"),
        # local Lagrangian density (baryons) from both potentials
        case("lla_uneven_o4", "lla", "128x192x160", order=4),
        # hybrid Poisson correction of a zoom's finest level
        case("hybrid_nest", "hybrid", "128x128x128", "128x96x112@30,41,35"),
        # the Gaussian density field itself, sides that are not powers of two
        case("field_uneven", "field", "192x200x243"),
    ]


def _side(rng, lo, hi, step):
    """A side in [lo, hi], spread over the logarithm, a multiple of step."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(step * int(math.ceil(lo / step)), step * int(v / step))


def _box(rng, lo, hi, order, ratio=4):
    """Sides of a periodic base, multiples of 4 that halve to a coarsest level of at most 4096
    cells, the longest at most ratio times the shortest."""
    while True:
        base = [_side(rng, lo, hi, 4) for _ in range(3)]
        n = list(base)
        while all(v % 2 == 0 for v in n) and max(n) > 8 and min(n) // 2 >= order // 2:
            n = [v // 2 for v in n]
        if max(base) <= ratio * min(base) and n[0] * n[1] * n[2] <= 4096:
            return base


def _nests(rng, base, order, count):
    text, parent = [], list(base)
    for _ in range(count):
        n, off = [], []
        for a in range(3):
            most = 2 * (parent[a] - 2 * order)
            side = 2 * int(rng.uniform(0.5, 1.0) * base[a] / 2)
            side = min(side, most - most % 2)
            n.append(side)
            off.append(rng.randint(order, parent[a] - side // 2 - order) if side >= 8 else 0)
        if min(n) < 8:
            break
        text.append("x".join(map(str, n)) + "@" + ",".join(map(str, off)))
        parent = n
    return ";".join(text)


def draw(rng):
    kind = rng.choice(["solve", "step", "step", "step", "step", "batch", "tau", "lla", "hybrid",
                       "field"])
    order = rng.choice([2, 4, 6, 6])
    mixed = rng.random() < 0.5
    c = {"kind": kind, "base": "", "nests": "", "order": order, "precision": "fp64", "tol": 3e-8,
         "inner": 4, "host": False, "members": 0}
    if kind in ("solve", "step"):
        while True:
            base = _box(rng, 32, 224, order)
            c["base"] = "x".join(map(str, base))
            c["nests"] = _nests(rng, base, order, rng.randint(0, 4))
            if _cells(c) <= ROOM:
                break
        c["precision"] = "mixed" if mixed else "fp64"
        c["inner"] = rng.choice([2, 3, 4])
        c["host"] = kind == "step" and rng.random() < 0.25
        c["tol"] = 1e-10 if kind == "solve" else 1e-8 if mixed else 3e-8
    elif kind == "batch":
        c.update(order=6, precision="mixed", tol=1e-8, members=rng.randint(4, 16))
    elif kind in ("tau", "lla"):
        c["base"] = "x".join(map(str, _box(rng, 32, 256, order, 8)))
    elif kind == "hybrid":
        base = _box(rng, 48, 128, order)
        c["base"] = "x".join(map(str, base))
        c["nests"] = _nests(rng, base, order, 1)
    else:
        c["base"] = "x".join(str(_side(rng, 31, 256, 1)) for _ in range(3))
    c["tag"] = rng.randrange(1 << 20) if kind == "batch" else 0
    return c


# ---- geometry ------------------------------------------------------------------------


def _base(case):
    return tuple(int(v) for v in case["base"].split("x"))


def _levels(case):
    """[(sides, origin in parent cells)], base first."""
    out = [(_base(case), (0, 0, 0))]
    for part in filter(None, case["nests"].split(";")):
        n, off = part.split("@")
        out.append((tuple(map(int, n.split("x"))), tuple(map(int, off.split(",")))))
    return out


def _members(case):
    """The geometries of a batch: bases of 32 to 96 cells a side, up to 3 nests."""
    import random
    rng = random.Random(4 + int(case.get("tag") or 0))
    out = []
    for _ in range(case["members"]):
        base = [rng.choice([32, 48, 64, 96])] * 3
        out.append(dict(case, base="x".join(map(str, base)),
                        nests=_nests(rng, base, case["order"], rng.randint(0, 3)), members=0))
    return out


def _cells(case):
    if case["members"]:
        return sum(_cells(m) for m in _members(case))
    return sum(n[0] * n[1] * n[2] for n, _ in _levels(case))


def _config(case):
    lv = _levels(case)
    return mg.make_config(lv[0][0], BOX, case["order"], lv[1:],
                          precision=mg.MG_MIXED if case["precision"] == "mixed" else mg.MG_FP64,
                          tol=case["tol"], inner_cycles=case["inner"])


# ---- inputs --------------------------------------------------------------------------


def _noise(gen, n):
    return torch.randn(n, generator=gen, device="cuda", dtype=torch.float64)


def _waves(n, h):
    """|k|^2 on the half spectrum of a periodic grid of spacing h."""
    k = [2 * math.pi * torch.fft.fftfreq(n[a], h, device="cuda", dtype=torch.float64)
         for a in range(2)]
    k.append(2 * math.pi * torch.fft.rfftfreq(n[2], h, device="cuda", dtype=torch.float64))
    return k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + k[2][None, None, :] ** 2


def _random_field(gen, n, h, power, rms):
    """A periodic Gaussian field of spectrum k^power and the given rms."""
    k2 = _waves(n, h)
    k2[0, 0, 0] = 1.0
    f = torch.fft.rfftn(_noise(gen, n)) * k2 ** (power / 4)
    f[0, 0, 0] = 0.0
    f = torch.fft.irfftn(f, s=n)
    return f * (rms / f.std())


def _densities(case, gen):
    lv = _levels(case)
    h = BOX / lv[0][0][0]
    out = [_random_field(gen, lv[0][0], h, -2.0, 0.05)]
    for n, off in lv[1:]:
        cut = out[-1][tuple(slice(o, o + s // 2) for o, s in zip(off, n))]
        up = torch.nn.functional.interpolate(cut[None, None], size=n, mode="trilinear")[0, 0]
        h /= 2
        out.append((up + _random_field(gen, n, h, -1.0, 0.03)).contiguous())
    return out


def _potential(gen, n, rms):
    return _random_field(gen, n, BOX / n[0], -6.0, rms)


def _outputs(shapes, host):
    """phi1, phi2 and both displacements of every level, as views of one allocation."""
    cells = [s[0] * s[1] * s[2] for s in shapes]
    flat = torch.empty(8 * sum(cells), dtype=torch.float64, pin_memory=host,
                       device="cpu" if host else "cuda")
    at, out = 0, {}
    for key, per in (("phi1", 1), ("phi2", 1), ("disp1", 3), ("disp2", 3)):
        out[key] = []
        for s, c in zip(shapes, cells):
            for _ in range(per):
                out[key].append(flat[at:at + c].view(s))
                at += c
    return flat, out


def _amplitude(nt, dk):
    """sqrt(P) of a spectrum that turns over at k = 0.02 and falls as k^-3."""
    k = np.arange(nt) * dk
    return np.sqrt(2e4 * (k / 0.02) / (1.0 + (k / 0.02) ** 2) ** 2)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind = case["kind"]
    if kind == "batch":
        members = [mg.Hierarchy(_config(m)) for m in _members(case)]
        deltas = [_densities(m, gen) for m in _members(case)]
        flat, outs = zip(*[_outputs(m.shapes, False) for m in members])
        return {"kind": kind, "batch": mg.Batch(members), "deltas": deltas, "outs": list(outs),
                "flat": list(flat)}
    if kind == "field":
        n = _base(case)
        h = BOX / n[0]
        nt, dk = 1024, math.pi / h * math.sqrt(3.0) / 1000
        return {"kind": kind, "seed": seed, "field": mg.Field(n, h, _amplitude(nt, dk), dk)}
    hier = mg.Hierarchy(_config(case))
    state = {"kind": kind, "h": hier, "host": case["host"]}
    n = _levels(case)[-1][0]
    if kind == "tau":
        state["phi"] = [_potential(gen, n, 40.0)]
    elif kind == "lla":
        # second derivatives of about 0.05: no shell crossing
        state["phi"] = [_potential(gen, n, 10.0)]
        state["phi2"] = [_potential(gen, n, 2.0)]
    elif kind == "hybrid":
        state["f"] = _densities(case, gen)[-1]
    else:
        state["delta"] = _densities(case, gen)
        if case["host"]:
            state["delta"] = [d.cpu().pin_memory() for d in state["delta"]]
        if kind == "step":
            state["outs"] = _outputs(hier.shapes, case["host"])[1]
    return state


def run(state):
    kind = state["kind"]
    if kind == "solve":
        phi, _ = state["h"].solve_1lpt(state["delta"])
        return phi
    if kind == "step":
        return state["h"].pipeline(state["delta"], state["outs"], host=state["host"])[0]
    if kind == "batch":
        state["batch"].pipeline(state["deltas"], state["outs"])
        return state["flat"]
    if kind == "tau":
        return state["h"].lpt2_source(state["phi"])
    if kind == "lla":
        return state["h"].lla_density(state["phi"], state["phi2"], 1.0, 0.4)
    if kind == "hybrid":
        psi = [torch.zeros_like(state["f"]) for _ in range(3)]
        return state["h"].hybrid_correction(state["f"], psi)
    return state["field"].generate(state["seed"])


# ---- what a pass cannot do without ---------------------------------------------------


def work(case):
    """Inputs read and outputs written once; operations of the method: per cell of a solve,
    V-cycles of four half-sweep pairs, residual and norm at about 2 (3 order + 1) operations
    each (a cycle takes the residual down by about 13; coarser levels add 1/7)."""
    c = _cells(case)
    o = case["order"]
    stencil = 3 * o + 2
    if case["kind"] in ("solve", "step", "batch"):
        cycles = math.ceil(math.log(1 / case["tol"]) / math.log(13.0))
        solve = cycles * 6 * stencil * c * 8 / 7
        if case["kind"] == "solve":
            return {"bytes": 16 * c, "flops": solve}
        return {"bytes": 72 * c, "flops": 2 * solve + 14 * stencil * c / 2}
    if case["kind"] == "tau":
        return {"bytes": 16 * c, "flops": 7 * o * c}
    if case["kind"] == "lla":
        return {"bytes": 24 * c, "flops": (7 * o + 20) * c}
    if case["kind"] == "hybrid":
        n = _levels(case)[-1][0]
        cells = n[0] * n[1] * n[2]
        return {"bytes": 7 * 8 * cells, "flops": 4 * 2.5 * 8 * cells * math.log2(8 * cells)}
    return {"bytes": 8 * c, "flops": 2 * 2.5 * c * math.log2(c) + 60 * c}


# ---- the same in plain 64-bit torch --------------------------------------------------

LAP = {2: (-2.0, 1.0), 4: (-30 / 12, 16 / 12, -1 / 12),
       6: (-490 / 180, 270 / 180, -27 / 180, 2 / 180)}
GRAD = {2: (0.5,), 4: (8 / 12, -1 / 12), 6: (45 / 60, -9 / 60, 1 / 60)}


def _shift(u, s, a):
    return torch.roll(u, -s, a)


def _second(u, a, order, h):
    w = LAP[order]
    return sum((w[s] * (_shift(u, s, a) + _shift(u, -s, a)) for s in range(1, len(w))),
               w[0] * u) / h ** 2


def _first(u, a, order, h):
    return sum(w * (_shift(u, s, a) - _shift(u, -s, a))
               for s, w in enumerate(GRAD[order], 1)) / h


def _inverse(f, order, h):
    """The zero-mean solution of the finite-difference Poisson equation, by Fourier."""
    lam = 0.0
    for a, n in enumerate(f.shape):
        m = n if a < 2 else n // 2 + 1
        t = 2 * math.pi * torch.arange(m, device="cuda", dtype=torch.float64) / n
        w = LAP[order]
        v = w[0] + sum(2 * w[s] * torch.cos(s * t) for s in range(1, len(w)))
        lam = lam + v.reshape([-1 if b == a else 1 for b in range(3)])
    lam[0, 0, 0] = 1.0
    F = torch.fft.rfftn(f - f.mean()) * (h * h) / lam
    F[0, 0, 0] = 0.0
    return torch.fft.irfftn(F, s=f.shape)


def _hessian(u, order, h):
    d = [_second(u, a, order, h) for a in range(3)]
    g = [_first(u, a, order, h) for a in range(3)]
    return d, [_first(g[b], a, order, h) for a, b in ((0, 1), (0, 2), (1, 2))]


def _tau(u, order, h):
    d, m = _hessian(u, order, h)
    return d[0] * d[1] + d[0] * d[2] + d[1] * d[2] - m[0] ** 2 - m[1] ** 2 - m[2] ** 2


def _exact_hybrid(f, order, h):
    """i [k_j / k^2 + g_j / L] f on the zero-padded grid, its Nyquist plane along j left out."""
    N = [2 * s for s in f.shape]
    F = torch.fft.rfftn(f, s=N)
    t, lam, g = [], 0.0, []
    for a in range(3):
        i = torch.arange(N[a] if a < 2 else N[a] // 2 + 1, device="cuda", dtype=torch.float64)
        ta = 2 * math.pi * torch.where(i <= N[a] // 2, i, i - N[a]) / N[a]
        shape = [-1 if b == a else 1 for b in range(3)]
        w = LAP[order]
        lam = lam + (w[0] + sum(2 * w[s] * torch.cos(s * ta) for s in range(1, len(w)))).reshape(shape)
        g.append(sum(2 * v * torch.sin(s * ta) for s, v in enumerate(GRAD[order], 1)).reshape(shape))
        t.append(ta.reshape(shape))
    k2 = t[0] ** 2 + t[1] ** 2 + t[2] ** 2
    k2[0, 0, 0] = 1.0
    lam[0, 0, 0] = 1.0
    out = []
    for a in range(3):
        c = h * (t[a] / k2 + g[a] / lam)
        c = torch.where(t[a].abs() > math.pi * (1 - 1e-12), torch.zeros_like(c), c)
        c[0, 0, 0] = 0.0
        out.append(torch.fft.irfftn(1j * c * F, s=N)[tuple(slice(0, s) for s in f.shape)].contiguous())
    return out


def _philox_normals(seed, n):
    """Philox4x32-10 and Box-Muller, as the library's header defines its white noise."""
    q = np.arange((n + 1) // 2, dtype=np.uint64)
    low = np.uint64(0xFFFFFFFF)
    s32 = np.uint64(32)
    x = [q & low, q >> s32, np.zeros_like(q), np.zeros_like(q)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
        p0, p1 = np.uint64(0xD2511F53) * x[0], np.uint64(0xCD9E8D57) * x[2]
        x = [(p1 >> s32) ^ x[1] ^ np.uint64(k0), p1 & low, (p0 >> s32) ^ x[3] ^ np.uint64(k1),
             p0 & low]

    def uniform(a, b):
        return ((a >> np.uint64(5)).astype(np.float64) * 2.0 ** 26
                + (b >> np.uint64(6)).astype(np.float64) + 0.5) / 2.0 ** 53

    r = np.sqrt(-2.0 * np.log(uniform(x[0], x[1])))
    t = 2.0 * np.pi * uniform(x[2], x[3])
    return np.stack([r * np.cos(t), r * np.sin(t)], 1).reshape(-1)[:n]


def exact(case, seed):
    """Closed forms exist where the grid is one periodic level.  The composite solution of
    a nested hierarchy has none, and a plain 64-bit solver for it takes minutes."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind, order = case["kind"], case["order"]
    if kind == "batch" or (kind in ("solve", "step") and case["nests"]):
        return None
    n = _levels(case)[-1][0]
    h = BOX / _base(case)[0]
    if kind == "tau":
        return [_tau(_potential(gen, n, 40.0), order, h)]
    if kind == "lla":
        u = _potential(gen, n, 10.0)
        u = u + 0.4 * _potential(gen, n, 2.0)
        d, m = _hessian(u, order, h)
        a, b, c = 1 - d[0], 1 - d[1], 1 - d[2]
        det = a * b * c - a * m[2] ** 2 - b * m[1] ** 2 - c * m[0] ** 2 - 2 * m[0] * m[1] * m[2]
        rho = 1.0 / det
        return [rho - rho.mean() + 1.0]
    if kind == "hybrid":
        return _exact_hybrid(_densities(case, gen)[-1], order, h / 2 ** (len(_levels(case)) - 1))
    if kind == "field":
        noise = torch.from_numpy(_philox_normals(seed, n[0] * n[1] * n[2]).reshape(n)).cuda()
        nt, dk = 1024, math.pi / h * math.sqrt(3.0) / 1000
        amp = torch.from_numpy(_amplitude(nt, dk)).cuda()
        t = torch.sqrt(_waves(n, h)) / dk
        i = t.floor().clamp(max=nt - 2).long()
        a = torch.where(t <= nt - 1, amp[i] + (t - i) * (amp[i + 1] - amp[i]), 0.0 * t)
        a[0, 0, 0] = 0.0
        return torch.fft.irfftn(torch.fft.rfftn(noise) * a, s=n)
    delta = _densities(case, gen)[0]
    phi1 = _inverse(delta, order, h)
    if kind == "solve":
        return [phi1]
    phi2 = _inverse(_tau(phi1, order, h), order, h)
    grads = [[-_first(p, a, order, h) for a in range(3)] for p in (phi1, phi2)]
    return {"phi1": [phi1], "phi2": [phi2], "disp1": grads[0], "disp2": grads[1]}
