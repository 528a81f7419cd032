"""What a user of this library has it do, as timed cases: whole solves and their state I/O.

A case is one pass through the public calls of ``paper_2512_16230_gb300.lbm`` the way a program that
solves a flow makes them: hand the initial fields over (device tensors), advance, read the fields
back. Three shapes of use exist and all are here:

* ``solve``       one model: ``init_fields``, ``step(steps)``, ``read_fields``;
* ``batch``       many models of a serving mix advanced together: ``Batch.step`` between the same calls;
* ``checkpoint``  a saved state taken up again: ``set_populations``, ``step``, the conservation sums,
                  ``get_populations``.

The lattices, flows, grids and storage types are those of the library's own workloads (the 2D vortex
and the nonlinear convection-diffusion hill, the 3D Taylor-Green vortex and the forced Kolmogorov flow;
32..1024 x 32..768 cells in 2D, 32..256 cells a side in 3D). Every field carries seeded noise, as a
flow taken up in mid-course does. Field I/O of the library is FP64; what a solve computes in FP32 or
stores in 16 bits is handed on in that type, since it holds no more.
"""
import itertools
import math

import numpy as np
import torch

from paper_2512_16230_gb300 import lbm

# name: (kind, axis speeds, squared sound speeds, free weights)
LATTICES = {
    "rD2Q25": ("rD2Q25", (1.0, 4 / 3), (0.8, 0.8), (3.125e-4,) * 4),
    "rD2Q21": ("rD2Q21", (1.0, 4 / 3), (0.8, 0.8), (7.29e-4,) * 3),
    "rD2Q17": ("rD2Q17", (1.0, 4 / 3), (0.8, 0.8), (2.1875e-3,)),
    "rD2Q13": ("rD2Q13", (1.0, 1.25), (0.8, 0.8), ()),
    "rD3Q53": ("rD3Q53", (1.0, 1.0, 4 / 3), (0.96, 0.96, 1.28), (8e-4,)),
    "rD3Q53-cubic": ("rD3Q53", (1.0, 1.0, 1.0), (0.6,) * 3, (2.4e-4,)),
    "rD3Q45": ("rD3Q45", (1.0, 1.0, 1.0), (0.6,) * 3, ()),
    "rD3Q33": ("rD3Q33", (1.0, 1.0, 1.0), (0.5,) * 3, ()),
}
ORDER_RATES = (0.9, 1.35, 1.6, 0.9, 1.25)  # rates of the orders 4..8 of the "order rates" option
RESULT = {"f64": torch.float64, "f32": torch.float32, "f16_dev": torch.float16, "bf16_dev": torch.bfloat16}
BYTES = {"f64": 8, "f32": 4, "f16_dev": 2, "bf16_dev": 2}
DEVICE = "cuda"
LARGEST = 256 * 256 * 192


def _solve(name, lattice, flow, n, steps, store="f32", rates=False):
    n = tuple(n) + (1,) * (3 - len(n))
    return dict(name=name, use="solve", lattice=lattice, flow=flow, nx=n[0], ny=n[1], nz=n[2], steps=steps,
                store=store, order_rates=rates)


def listed():
    return [
        # the smallest served request: a 2D vortex whose step is a few microseconds
        _solve("vortex2d-small", "rD2Q17", "vortex", (64, 48), 100),
        # the decaying vortex used to verify a set-up, in double precision
        _solve("vortex2d-f64", "rD2Q25", "vortex", (64, 48), 100, "f64"),
        # a mid-size served scalar transport problem with odd extents
        _solve("hill2d-odd", "rD2Q21", "hill", (413, 295), 100),
        # nonlinear convection-diffusion on the 1024 x 768 grid
        _solve("hill2d-large", "rD2Q13", "hill", (1024, 768), 100),
        # forced 3D flow of the serving mix, mid size
        _solve("kolmogorov-64", "rD3Q33", "kolmogorov", (64, 64, 64), 64),
        # the same flow where no extent is a multiple of anything
        _solve("kolmogorov-odd", "rD3Q45", "kolmogorov", (101, 103, 97), 32),
        # the 3D Taylor-Green vortex at full size, single precision
        _solve("vortex3d-f32", "rD3Q53", "vortex", (256, 256, 192), 24),
        # the same with FP16 deviations as storage
        _solve("vortex3d-f16", "rD3Q53", "vortex", (256, 256, 192), 24, "f16_dev"),
        # BF16 storage on a ragged grid
        _solve("kolmogorov-bf16-odd", "rD3Q53-cubic", "kolmogorov", (150, 131, 147), 24, "bf16_dev"),
        # one relaxation rate per order (the full collision), single precision
        _solve("vortex3d-rates", "rD3Q53", "vortex", (160, 144, 120), 24, "f32", True),
        # a serving mix advanced together: small and large, 2D and 3D
        dict(name="batch-mix", use="batch", solves=24, mix=1, steps=64, store="f32"),
        # a state written out and taken up again
        dict(_solve("checkpoint", "rD3Q53", "vortex", (128, 128, 96), 8), use="checkpoint"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    most = max(work(c)["bytes"] for c in listed())
    while True:  # a drawn case costs no more than the largest listed one
        case = _draw(rng)
        if work(case)["bytes"] <= most:
            return case


def _draw(rng):
    use = rng.choice(["2d", "2d", "3d", "3d", "3d", "batch", "checkpoint"])
    if use == "batch":
        return dict(use="batch", solves=rng.randint(6, 24), mix=rng.randrange(1 << 20), steps=rng.randint(16, 64),
                    store=rng.choice(["f32", "f32", "f16_dev"]))
    if use == "2d":
        flow = rng.choice(["vortex", "hill"])
        lattice = rng.choice(["rD2Q13", "rD2Q17", "rD2Q21", "rD2Q25"])
        store = rng.choice(["f32", "f32", "f32", "f64", "f16_dev"])
        return {k: v for k, v in _solve("", lattice, flow, (_log(rng, 32, 1024), _log(rng, 32, 768)),
                                        rng.randint(50, 100), store).items() if k != "name"}
    lattice = rng.choice(["rD3Q33", "rD3Q45", "rD3Q53-cubic", "rD3Q53"])
    flow = "vortex" if lattice == "rD3Q53" else "kolmogorov"
    store = rng.choice(["f32", "f32", "f16_dev", "bf16_dev"])
    n = [_log(rng, 32, 256) for _ in range(3)]
    if rng.random() < 0.5:  # rows of whole 16-byte pieces, as grids are usually chosen
        n[0] = max(32, n[0] // 8 * 8)
    while n[0] * n[1] * n[2] > LARGEST:
        n[rng.randint(1, 2)] //= 2
    if use == "checkpoint":
        n[2] = max(8, min(n[2], 128 * 128 * 96 // (n[0] * n[1])))
        c = _solve("", lattice, flow, n, rng.randint(1, 8), store)
        return {k: v for k, v in dict(c, use="checkpoint").items() if k != "name"}
    c = _solve("", lattice, flow, n, rng.randint(8, 24), store, rng.random() < 0.25)
    return {k: v for k, v in c.items() if k != "name"}


# --- the problems -----------------------------------------------------------------------------

def _members(case):
    """The solves of a case: one, or the seeded mix of a batch (half 2D, half forced 3D)."""
    if case["use"] != "batch":
        return [case]
    rng = np.random.default_rng(case["mix"])
    out = []
    for k in range(case["solves"]):
        lg = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
        if k % 2:
            lattice, flow, side = ("rD3Q33", "rD3Q45", "rD3Q53-cubic")[int(rng.integers(3))], "kolmogorov", lg(32, 112)
            n = (side, side, side)
        else:
            lattice, flow = ("rD2Q17", "rD2Q21", "rD2Q25")[int(rng.integers(3))], ("vortex", "hill")[int(rng.integers(2))]
            n = (lg(32, 1024), lg(32, 768), 1)
        out.append(dict(lattice=lattice, flow=flow, nx=n[0], ny=n[1], nz=n[2], steps=case["steps"],
                        store=case["store"], order_rates=False))
    return out


def _problem(m):
    """Grid, rates, force and base amplitude of one solve."""
    kind, c, cs2, _ = LATTICES[m["lattice"]]
    d = len(c)
    n = (m["nx"], m["ny"], m["nz"])[:d]
    orders = [0, 1, 1] + [2] * 3 + [3] * 4 if d == 2 else [0, 1, 1, 1] + [2] * 6 + [3] * 10
    length = n[0] * c[0] / (2 * math.pi)
    p = dict(kind=kind, c=c, cs2=cs2, d=d, n=n, eq="ncde" if m["flow"] == "hill" else "nse", force=None, u_const=None)
    if m["flow"] == "hill":
        p.update(s1=1 / (0.1 / cs2[0] + 0.5), s2=1.0, u_const=(0.02, 0.01), nonlin=1.0)
    else:
        if m["flow"] == "kolmogorov":
            u0, nu = 0.05 * math.sqrt(cs2[0]), 0.05
            p["force"] = (0, 1, u0 * nu * (2 * math.pi / (n[1] * c[1])) ** 2)
        elif d == 2:
            u0 = 0.05 * math.sqrt(cs2[0])
            nu = u0 * length / 100
        else:
            u0 = 0.3 * math.sqrt(cs2[0])
            nu = u0 * length / 1600
        p.update(s1=1.0, s2=1 / (nu / cs2[0] + 0.5), u0=u0)
    p["s"] = [p["s1"] if o == 1 else p["s2"] if o == 2 else 1.0 for o in orders]
    p["rates"] = ORDER_RATES if m["order_rates"] else ()
    return p


def _fields(m, p, seed):
    """Initial fields on the GPU, (rho, u) or (phi, None): the flow's own and seeded noise on it."""
    g = torch.Generator(device=DEVICE).manual_seed(seed)
    d, n, c = p["d"], p["n"], p["c"]
    shape = tuple(reversed(n))
    ang = []
    for a in range(d):
        x = torch.arange(n[a], dtype=torch.float64, device=DEVICE) * (2 * math.pi / n[a])
        ang.append(x.reshape([-1 if b == d - 1 - a else 1 for b in range(d)]).expand(shape))
    noise = lambda *s: 2 * torch.rand(*s, generator=g, dtype=torch.float64, device=DEVICE) - 1  # noqa: E731
    if m["flow"] == "hill":
        sigma = max(2.0, n[0] / 8)
        r2 = sum(((ang[a] / (2 * math.pi) - 0.5) * n[a] * c[a]) ** 2 for a in range(d))
        return (torch.exp(-r2 / (2 * sigma ** 2)) + 1e-3 * noise(*shape)).contiguous(), None
    u0 = p["u0"]
    if m["flow"] == "kolmogorov":
        u = [u0 * torch.sin(ang[1]), 0 * ang[0], 0 * ang[0]]
        rho = torch.ones(shape, dtype=torch.float64, device=DEVICE)
    elif d == 2:
        kx, ky = 1 / (n[0] * c[0]), 1 / (n[1] * c[1])
        k = math.hypot(kx, ky) / math.sqrt(2)
        u = [-u0 * ky / k * torch.cos(ang[0]) * torch.sin(ang[1]), u0 * kx / k * torch.sin(ang[0]) * torch.cos(ang[1])]
        rho = 1 - 0.25 * u0 ** 2 / p["cs2"][0] * ((ky / k) ** 2 * torch.cos(2 * ang[0]) + (kx / k) ** 2 * torch.cos(2 * ang[1]))
    else:
        X, Y, Z = ang
        u = [u0 * torch.sin(X) * torch.cos(Y) * torch.cos(Z), -u0 * torch.cos(X) * torch.sin(Y) * torch.cos(Z), 0 * X]
        rho = 1 + u0 ** 2 / (16 * p["cs2"][0]) * (torch.cos(2 * X) + torch.cos(2 * Y)) * (torch.cos(2 * Z) + 2)
    return (rho + 1e-3 * noise(*shape)).contiguous(), torch.stack(u) + 0.02 * u0 * noise(d, *shape)


# --- the pass through the library ---------------------------------------------------------------

def _model(m, p, lattice):
    model = lbm.Model(lattice, p["eq"], p["n"], store=m["store"])
    model.set_relaxation(p["s"])
    if p["rates"]:
        model.set_high_rates(p["rates"])
    if p["force"]:
        model.set_force(*p["force"], 1)
    if p["u_const"]:
        model.set_ncde(p["u_const"], p["nonlin"])
    return model


def prepare(case, seed):
    state, lattices = dict(case=case, solves=[], batch=None), {}
    if case["use"] == "batch":
        state["batch"] = lbm.Batch()
        state["stream"] = torch.cuda.ExternalStream(state["batch"].stream)
    for k, m in enumerate(_members(case)):
        p = _problem(m)
        if m["lattice"] not in lattices:
            lattices[m["lattice"]] = lbm.Lattice(*LATTICES[m["lattice"]])
        model = _model(m, p, lattices[m["lattice"]])
        rho, u = _fields(m, p, seed + 7919 * k)
        s = dict(model=model, rho=rho, u=u, rho_out=torch.empty_like(rho),
                 u_out=None if u is None else torch.empty_like(u), dtype=RESULT[m["store"]])
        if case["use"] == "checkpoint":
            model.init_fields(rho, u)  # the state that was saved
            s["f"] = model.get_populations(torch.empty((model.Q,) + tuple(reversed(p["n"])), dtype=torch.float64, device=DEVICE))
            s["f_out"] = torch.empty_like(s["f"])
            s["sums"] = torch.zeros(4, dtype=torch.float64, device=DEVICE)
        if state["batch"] is not None:
            state["batch"].add(model)
        state["solves"].append(s)
    return state


def run(state):
    case, solves = state["case"], state["solves"]
    if case["use"] == "checkpoint":
        s = solves[0]
        m = s["model"]
        m.set_populations(s["f"])
        m.step(case["steps"])
        m.conserved_sums_noalloc(s["sums"])
        m.get_populations(s["f_out"])
        return {"f": s["f_out"].to(s["dtype"]), "sums": s["sums"].to(s["dtype"])}
    if state["batch"] is None:
        s = solves[0]
        s["model"].init_fields(s["rho"], s["u"])
        s["model"].step(case["steps"])
        return _read(s)
    batch, ext = state["batch"], state["stream"]
    ext.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(ext):
        for s in solves:
            s["model"].init_fields(s["rho"], s["u"])
        batch.step(case["steps"])
        out = [_read(s) for s in solves]
    torch.cuda.current_stream().wait_stream(ext)
    return out


def _read(s):
    s["model"].read_fields(s["rho_out"], s["u_out"])
    u = s["u_out"]
    return {"rho": s["rho_out"].to(s["dtype"]), "u": None if u is None else u.to(s["dtype"])}


def work(case):
    """Bytes: the initial fields in and the final fields out, and the populations once in and once out
    for each step (a step's whole input and output); flops: the two contractions with the rows of
    order <= 3, factored by velocity pairs, and the moment-space update, per cell and step."""
    total = dict(bytes=0, flops=0)
    for m in _members(case):
        kind, c, _, _ = LATTICES[m["lattice"]]
        d, q = len(c), int(kind[4:])
        r = 10 if d == 2 else 20
        cells = m["nx"] * m["ny"] * m["nz"]
        fields = 1 if m["flow"] == "hill" else 1 + d
        io = 2 * 8 * (q if case["use"] == "checkpoint" else fields)
        history = 2 * (8 if m["store"] == "f64" else 4) if m["flow"] == "hill" else 0
        total["bytes"] += cells * (io + m["steps"] * (2 * q * BYTES[m["store"]] + history))
        high = 4 * q * (q - r) // 2 if m["order_rates"] else 0
        total["flops"] += cells * m["steps"] * (2 * q * r // 2 + 4 * r * d + 6 * q + high)
    return total


# --- the same in 64 bits, written out plainly -----------------------------------------------------

def _velocities(kind):
    q = int(kind[4:])
    if kind.startswith("rD2"):
        axis = [(1, 0), (0, 1), (-1, 0), (0, -1)]
        diag = [(1, 1), (-1, 1), (-1, -1), (1, -1)]
        e = [(0, 0)] + [(m * x, m * y) for m in (1, 2, 3) for x, y in axis + diag]
        return np.array(e[:q], dtype=np.int64)
    one = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, 1), (0, 1, 1), (0, -1, 1),
           (1, 1, 1), (1, 1, -1), (1, -1, 1), (-1, 1, 1)]
    pairs = [v for x in one for v in (x, tuple(-t for t in x))]
    return np.array(([(0, 0, 0)] + pairs + [tuple(2 * t for t in v) for v in pairs])[:q], dtype=np.int64)


def _weights(kind, e, c, cs2, free):
    """One weight per reflection class: the free ones as given, the others from sum w = 1 and the
    lattice moments of a Gaussian, E[c_a^2] = s_a, E[c_a^4] = 3 s_a^2, E[c_a^2 c_b^2] = s_a s_b and in 3D
    E[c_x^2 c_y^2 c_z^2] and E[c_a^4 c_b^2] (a < b) (the weight conditions of the method)."""
    d, dd = len(c), np.array(cs2) / np.array(c) ** 2
    classes = sorted(set(map(tuple, np.abs(e))))
    fixed = {}
    if kind == "rD3Q53":
        fixed[(2, 2, 2)] = free[0]
    elif d == 2 and free:
        fixed = dict(zip([(2, 2), (3, 0), (0, 3), (3, 3)], free))
    gauss = [1.0, dd, 3 * dd ** 2]
    powers = [(0,) * d] + [p for p in itertools.product((0, 2, 4), repeat=d) if 0 < sum(p) <= 6]
    powers = [p for p in powers if 4 not in p or sum(p) == 4 or (d == 3 and sum(p) == 6)]
    powers = [p for p in powers if d == 3 or sum(p) <= 4]
    if d == 3:  # one of x^4 y^2 / x^2 y^4 for each pair of axes; none where the lattice has no such class
        powers = [p for p in powers if not (4 in p and 2 in p) or (p.index(4) < p.index(2) and kind != "rD3Q33")]
    unknown = [k for k in classes if k not in fixed]
    A, b = [], []
    for p in powers:
        mono = np.prod(e.astype(float) ** np.array(p), axis=1)
        by = {k: mono[(np.abs(e) == k).all(axis=1)].sum() for k in classes}
        A.append([by[k] for k in unknown])
        want = np.prod([gauss[q // 2][a] if q else 1.0 for a, q in enumerate(p)])
        b.append(want - sum(by[k] * v for k, v in fixed.items()))
    w = {**dict(zip(unknown, np.linalg.lstsq(np.array(A), np.array(b), rcond=None)[0])), **fixed}
    return np.array([w[tuple(k)] for k in np.abs(e)])


def _exact_solve(m, seed, populations=False):
    p = _problem(m)
    d, n, cs2 = p["d"], p["n"], p["cs2"]
    e = _velocities(p["kind"])
    w = _weights(p["kind"], e, p["c"], cs2, LATTICES[m["lattice"]][3])
    cv = e * np.array(p["c"])
    exps = lambda k: [x for x in itertools.product(range(k + 1), repeat=d) if sum(x) == k]  # noqa: E731
    mono = lambda x: np.prod(cv ** np.array(x), axis=1)  # noqa: E731
    # orthonormal functions of each order (inner product sum_i w_i g h), order by order
    sw, basis, blocks = np.sqrt(w), np.zeros((0, len(w))), []
    for k in range(9):
        new = []
        for x in exps(k):
            v = mono(x) * sw
            v = v / np.linalg.norm(v)
            for _ in range(2):
                for b in list(basis) + new:
                    v = v - (b @ v) * b
            if np.linalg.norm(v) > 1e-9:
                new.append(v / np.linalg.norm(v))
        blocks.append(np.array(new).reshape(-1, len(w)))
        basis = np.concatenate([basis, blocks[-1]])
    rate = [1.0, p["s1"], p["s2"], 1.0] + [p["rates"][k - 4] if k - 4 < len(p["rates"]) else 1.0 for k in range(4, 9)]
    relax = sum(s * (sw[:, None] * b.T) @ (b / sw) for s, b in zip(rate, blocks))  # acts on populations
    top = 2 if p["eq"] == "ncde" else 3
    keys = [x for k in range(top + 1) for x in exps(k)]
    B = np.array([mono(x) for x in keys])
    lift = (w * B).T @ np.linalg.inv(B @ (w[:, None] * B.T))  # populations with these raw moments, order <= top
    second = [x for x in exps(2)]
    H2 = np.array([mono(x) for x in second])
    low = np.concatenate(blocks[:2])
    H2 = H2 - (H2 * sw) @ low.T @ (low / sw)
    lift2 = (w * H2).T @ np.linalg.inv(H2 @ (w[:, None] * H2.T))
    lift1 = w[:, None] * cv / np.array(cs2)
    t = lambda v: torch.tensor(v, dtype=torch.float64, device=DEVICE)  # noqa: E731
    keep, gain, lift, lift1, lift2, C = t(np.eye(len(w)) - relax), t(relax @ lift), t(lift), t(lift1), t(lift2), t(cv.T.copy())
    rho, u = _fields(m, p, seed)
    shape, cells = rho.shape, rho.numel()

    def moments(r, v):  # raw moments of the equilibrium
        out = []
        for x in keys:
            ax = [a for a in range(d) for _ in range(x[a])]
            if p["eq"] == "ncde":
                D = r + p["nonlin"] * r ** 3 / 3
                out.append(r if not ax else p["u_const"][ax[0]] * r if len(ax) == 1 else
                           cs2[0] * D if ax[0] == ax[1] else torch.zeros_like(r))
                continue
            term = r.clone()
            for a in ax:
                term = term * v[a]
            if len(ax) == 2 and ax[0] == ax[1]:
                term = term + cs2[0] * r
            if len(ax) == 3:
                for i, j, k in ((0, 1, 2), (1, 0, 2), (2, 0, 1)):
                    if ax[j] == ax[k]:
                        term = term + cs2[0] * r * v[ax[i]]
            out.append(term)
        return torch.stack(out)

    rho, u = rho.reshape(-1), None if u is None else u.reshape(d, -1)
    F = None
    if p["force"]:
        a, b, A = p["force"]
        prof = A * torch.sin(torch.arange(n[b], dtype=torch.float64, device=DEVICE) * (2 * math.pi / n[b]))
        F = torch.zeros((d,) + tuple(shape), dtype=torch.float64, device=DEVICE)
        F[a] = prof.reshape([-1 if k == d - 1 - b else 1 for k in range(d)])
        F = F.reshape(d, -1)
    f = lift @ moments(rho, u)
    prev = rho

    def fields(f):
        r = f.sum(0)
        if p["eq"] == "ncde":
            return r, None
        j = C @ f
        return r, (j + 0.5 * F if F is not None else j) / r

    for _ in range(m["steps"]):
        r, v = fields(f)
        g = keep @ f
        del f
        g.addmm_(gain, moments(r, v))
        if F is not None:
            g.addmm_(lift1, (1 - p["s1"] / 2) * F)
            both = []
            for x in second:
                i, j = [a for a in range(d) for _ in range(x[a])]
                both.append((1 - p["s2"] / 2) * (v[i] * F[j] + v[j] * F[i]))
            g.addmm_(lift2, torch.stack(both))
        if p["eq"] == "ncde":
            g.addmm_(lift1, (1 - p["s1"] / 2) * torch.stack([k * (r - prev) for k in p["u_const"]]))
            prev = r
        g = g.reshape((len(w),) + tuple(shape))
        for i in range(len(w)):
            g[i] = torch.roll(g[i], tuple(int(x) for x in e[i]), dims=tuple(range(d - 1, -1, -1)))
        f = g.reshape(len(w), cells)
    if populations:
        sums = torch.zeros(4, dtype=torch.float64, device=DEVICE)
        sums[0] = f.sum()
        sums[1:1 + d] = (C @ f).sum(1)
        return {"f": f.reshape((len(w),) + tuple(shape)), "sums": sums}
    r, v = fields(f)
    return {"rho": r.reshape(shape), "u": None if v is None else v.reshape((d,) + tuple(shape))}


def exact(case, seed):
    if case["use"] == "checkpoint":
        # the sums of a 16-bit state have no value of their own: the momentum in them is rounding
        out = _exact_solve(case, seed, True)
        return {"f": out["f"], "sums": out["sums"] if case["store"] in ("f32", "f64") else None}
    outs = [_exact_solve(m, seed + 7919 * k) for k, m in enumerate(_members(case))]
    return outs if case["use"] == "batch" else outs[0]
