"""The work a user of the library has it do, as cases that can be timed.

Every case goes through the package's public entry points.  Most are jobs: a
field that the user holds is loaded into a lattice's state and relaxed for a
while; the rest are the passes a run starts or ends with (seeding, energy,
observables, a picture).  ``prepare`` makes what the user has in hand, ``run``
is one pass, ``exact`` the same results from plain 64-bit torch.

Fields are product-ansatz clusters of 1-Skyrmions (Section 4.2) or smoothed
noise, as in ``workloads``, with positions, orientations and noise drawn from
the seed.  Flows return the updated state (field and velocity) and their report.
"""
import math

import numpy as np
import torch

import paper_2604_25876_gb300 as sk

DEV = "cuda"
MODES = {"arrested": sk.ARRESTED, "newton": sk.NEWTON, "gradient": sk.GRADIENT}


# ------------------------------------------------------------------ cases
def flow(name, entry, precision, n, h, steps, B, radius, m=1.0, m_w=0.0, c6=0.0, mode="arrested",
         courant=0.05, scale=1.0):
    c = {"name": name, "kind": "flow", "entry": entry, "precision": precision, "n0": n[0],
         "n1": n[1], "n2": n[2], "h": h, "m": m, "m_w": m_w, "c6": c6, "mode": mode,
         "steps": steps, "B": B, "radius": radius, "scale": scale, "dt": courant * h}
    return c


def listed():
    return [
        # one iteration at a time with its report on a small lattice, as an
        # interactive program or a test steps it: latency counts
        flow("f32_single_step_24", "step", 32, (24, 26, 28), 0.25, 1, 1, 0.3),
        # the benchmark's end-to-end job: 128^3 from and to pinned host memory
        flow("f32_host_job_128", "host", 32, (128, 128, 128), 0.1, 20, 4, 2.0),
        # a production relaxation: 256^3 cluster, iterations replayed as a graph
        flow("f32_graph_256", "graph", 32, (256, 256, 256), 0.08, 20, 8, 3.0),
        # the largest configured lattice
        flow("f32_flow_512", "step", 32, (512, 512, 512), 0.06, 4, 32, 6.0, courant=0.025),
        # an extended model (sextic term) on a lattice with odd sides, plain Newton flow
        flow("f32_sextic_odd", "step", 32, (113, 125, 107), 0.1, 20, 2, 1.5, c6=1.0, mode="newton",
             courant=0.0125, scale=2.0),
        # many stochastic starts of uneven sizes in one persistent launch
        {"name": "f32_batch_16", "kind": "batch", "count": 16, "low": 64, "high": 128, "h": 0.15,
         "m": 1.0, "dt": 0.0075, "steps": 50, "radius": 3.0, "sigma": 1.0},
        # the massless hedgehog workload in FP64
        flow("f64_flow_48", "step", 64, (48, 48, 48), 0.2, 25, 1, 0.3, m=0.0),
        # FP64 relaxation of a lightly bound model on a ragged lattice
        flow("f64_lightly_bound_ragged", "step", 64, (90, 75, 83), 0.15, 10, 3, 2.0, m_w=1.0),
        # energy, charge and virial of a relaxed-size FP32 field
        {"name": "energy_f32_256", "kind": "energy", "precision": 32, "n0": 256, "n1": 256,
         "n2": 256, "h": 0.08, "m": 1.0, "B": 8, "radius": 3.0},
        # the Section 5 observables on the paper's default lattice
        {"name": "observables_f32_151", "kind": "observables", "precision": 32, "n0": 151,
         "n1": 151, "n2": 151, "h": 16.0 / 150.0, "m": 1.0, "B": 4, "radius": 2.0},
        # a picture of the 128^3 field
        {"name": "render_f32_128", "kind": "render", "precision": 32, "n0": 128, "n1": 128,
         "n2": 128, "h": 0.1, "m": 1.0, "B": 4, "radius": 2.0, "width": 1024, "height": 768,
         "step": 0.005, "levelset": 0.2},
        # seeding the 256^3 cluster workload
        {"name": "seed_cluster_256", "kind": "seed", "precision": 32, "n0": 256, "n1": 256,
         "n2": 256, "h": 0.08, "m": 1.0, "B": 8, "radius": 3.0, "symmetrise": True},
    ]


def draw(rng):
    def side(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def box(lo, hi):
        return {"n0": side(lo, hi), "n1": side(lo, hi), "n2": side(lo, hi)}

    kind = rng.choice(["flow32", "flow32", "flow32", "flow64", "flow64", "batch", "energy",
                       "observables", "render", "seed"])
    if kind in ("flow32", "flow64"):
        p = 32 if kind == "flow32" else 64
        nn = box(20, 288) if p == 32 else box(20, 128)
        h = rng.uniform(0.1, 0.25)
        model = rng.choice(["standard", "standard", "lightly", "sextic"])
        return dict({"kind": "flow", "entry": rng.choice(["step", "graph", "host"]),
                     "precision": p, "h": h, "m": rng.choice([0.0, 1.0]),
                     "m_w": 1.0 if model == "lightly" else 0.0,
                     "c6": 1.0 if model == "sextic" else 0.0,
                     "mode": rng.choice(["arrested", "arrested", "newton", "gradient"]),
                     "steps": rng.choice([1, 2, 5, 10, 20]),
                     "B": rng.choice([1, 2] if model == "sextic" else [1, 2, 4]),
                     "radius": min(2.0, 0.2 * h * min(nn.values())),
                     # the sextic term is stiff on steep profiles
                     "scale": 2.0 if model == "sextic" else 1.0,
                     "dt": (0.0125 if model == "sextic" else 0.025) * h}, **nn)
    if kind == "batch":
        low = rng.randint(24, 96)
        return {"kind": "batch", "count": rng.randint(2, 24), "low": low,
                "high": rng.randint(low, 128), "h": 0.15, "m": 1.0, "dt": 0.0075,
                "steps": rng.choice([2, 10, 20]), "radius": rng.uniform(1.0, 3.0), "sigma": 1.0}
    p = rng.choice([32, 32, 64])
    if kind == "energy":
        nn, h = box(24, 288), rng.uniform(0.08, 0.2)
        return dict({"kind": "energy", "precision": p, "h": h, "m": rng.choice([0.0, 1.0]),
                     "B": rng.choice([1, 2, 8]), "radius": min(3.0, 0.2 * h * min(nn.values()))},
                    **nn)
    if kind == "observables":
        nn, h = box(24, 180), rng.uniform(0.1, 0.2)
        return dict({"kind": "observables", "precision": p, "h": h, "m": 1.0,
                     "B": rng.choice([2, 3, 4]), "radius": min(2.0, 0.2 * h * min(nn.values()))},
                    **nn)
    if kind == "render":
        nn, h = box(32, 160), rng.uniform(0.1, 0.2)
        return dict({"kind": "render", "precision": p, "h": h, "m": 1.0, "B": rng.choice([1, 4]),
                     "radius": min(2.0, 0.2 * h * min(nn.values())), "width": rng.randint(64, 1024),
                     "height": rng.randint(48, 768), "step": rng.uniform(0.005, 0.02),
                     "levelset": rng.uniform(0.05, 0.5)}, **nn)
    nn, h = box(24, 256), rng.uniform(0.08, 0.2)
    return dict({"kind": "seed", "precision": p, "h": h, "m": 1.0, "B": rng.randint(1, 8),
                 "radius": min(3.0, 0.25 * h * min(nn.values())),
                 "symmetrise": rng.choice([True, False])}, **nn)


# ----------------------------------------------------------------- inputs
def sizes(case):
    return (case["n0"], case["n1"], case["n2"])


def lattice(case, n=None):
    return sk.Lattice(n or sizes(case), case["h"], case["m"], case.get("precision", 32),
                      m_w=case.get("m_w", 0.0), c6=case.get("c6", 0.0))


def constituents(case, seed):
    """Seeded positions in a ball and iso-orientations (unit quaternions)."""
    rng = np.random.default_rng(seed)
    pos = []
    while len(pos) < case["B"]:
        p = rng.uniform(-case["radius"], case["radius"], size=3)
        if p @ p <= case["radius"] ** 2:
            pos.append(p)
    q = rng.normal(size=(case["B"], 4))
    return np.array(pos), q / np.linalg.norm(q, axis=1, keepdims=True)


def quat_mul(a, b):
    """Product of SU(2) elements a0 + i a.tau as lists of 4 tensors or numbers."""
    return [a[0] * b[0] - (a[1] * b[1] + a[2] * b[2] + a[3] * b[3]),
            a[0] * b[1] + b[0] * a[1] - (a[2] * b[3] - a[3] * b[2]),
            a[0] * b[2] + b[0] * a[2] - (a[3] * b[1] - a[1] * b[3]),
            a[0] * b[3] + b[0] * a[3] - (a[1] * b[2] - a[2] * b[1])]


def product_field(n, h, pos, quat, dtype, scale=1.0, symmetrise=False, x0=0, x1=None):
    """Product ansatz U_1 .. U_K of isorotated hedgehogs f = pi exp(-r / scale) on
    the planes x0 .. x1, shape (x1 - x0, n1, n2, 4)."""
    x1 = n[0] if x1 is None else x1
    ax = [(torch.arange(a, b, dtype=torch.float64, device=DEV) - 0.5 * (m - 1)) * h
          for a, b, m in ((x0, x1, n[0]), (0, n[1], n[1]), (0, n[2], n[2]))]
    shape = [(-1, 1, 1), (1, -1, 1), (1, 1, -1)]
    fwd = rev = None
    for p, q in zip(pos, quat):
        d = [(ax[i] - float(p[i])).to(dtype).reshape(shape[i]) for i in range(3)]
        r = torch.sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2])
        f = math.pi * torch.exp(-r / scale)
        s = torch.sin(f) / torch.where(r > 0, r, torch.ones_like(r))
        u = [torch.cos(f), s * d[0], s * d[1], s * d[2]]
        a = [float(v) for v in q]
        u = quat_mul(quat_mul(a, u), [a[0], -a[1], -a[2], -a[3]])
        fwd, rev = (u, u) if fwd is None else (quat_mul(fwd, u), quat_mul(u, rev) if symmetrise
                                               else None)
    out = [x + y for x, y in zip(fwd, rev)] if symmetrise else fwd
    norm = torch.sqrt(out[0] ** 2 + out[1] ** 2 + out[2] ** 2 + out[3] ** 2)
    if symmetrise:
        small = norm < 1e-12
        return torch.stack([torch.where(small, g, v / norm) for g, v in zip(fwd, out)], -1)
    return torch.stack([v / norm for v in out], -1) if dtype == torch.float32 else torch.stack(out, -1)


def cluster_field(case, seed):
    dtype = torch.float64 if case["precision"] == 64 else torch.float32
    pos, quat = constituents(case, seed)
    return product_field(sizes(case), case["h"], pos, quat, dtype, case.get("scale", 1.0))


def batch_sides(case, seed):
    rng = np.random.default_rng(4)  # the same mixture of sizes for every seed
    return [int(v) for v in rng.integers(case["low"], case["high"] + 1, size=case["count"])]


def noise_field(case, side, seed):
    """Vacuum plus Gaussian-smoothed normal noise from a ball, normalised."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    h, sigma = case["h"], case["sigma"]
    x = (torch.arange(side, dtype=torch.float32, device=DEV) - 0.5 * (side - 1)) * h
    ball = (x.reshape(-1, 1, 1) ** 2 + x.reshape(1, -1, 1) ** 2 + x.reshape(1, 1, -1) ** 2
            <= case["radius"] ** 2)
    v = torch.randn((side, side, side, 4), generator=g, device=DEV) * ball[..., None]
    w = torch.exp(-((x[:, None] - x[None, :]) ** 2) / (2 * sigma ** 2))
    w = w * ((x[:, None] - x[None, :]).abs() <= 4 * sigma)
    for eq in ("ax,xyzc->ayzc", "by,xyzc->xbzc", "cz,xyzd->xycd"):
        v = torch.einsum(eq, w, v)
    v = v / v[ball].std(dim=0)
    v[..., 0] += 1.0
    return v / v.norm(dim=-1, keepdim=True)


def render_view(seed):
    q = np.random.default_rng(seed).normal(size=4)
    a, b, c, d = q / np.linalg.norm(q)
    return np.array([[a * a + b * b - c * c - d * d, 2 * (b * c - a * d), 2 * (b * d + a * c)],
                     [2 * (b * c + a * d), a * a - b * b + c * c - d * d, 2 * (c * d - a * b)],
                     [2 * (b * d - a * c), 2 * (c * d + a * b), a * a - b * b - c * c + d * d]])


# ---------------------------------------------------------- prepare and run
def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        sides = batch_sides(case, seed)
        lats = [lattice(case, (N, N, N)) for N in sides]
        states = [sk.State(lat, DEV) for lat in lats]
        fields = [noise_field(case, N, 1000 * seed + k) for k, N in enumerate(sides)]
        for lat, st, phi in zip(lats, states, fields):
            sk.load_field(lat, st, phi)
        batch = sk.Batch(lats, states, [case["dt"]] * len(lats), sk.ARRESTED)
        batch.set_tile(4)  # the tile the autotuner picks for the batched workload
        return {"case": case, "batch": batch, "fields": fields}
    lat = lattice(case)
    st = sk.State(lat, DEV)
    s = {"case": case, "lat": lat, "st": st}
    if kind == "seed":
        pos, quat = constituents(case, seed)
        s["seed"] = sk.Seed.product(pos, quat, 1.0, case["symmetrise"])
        return s
    s["phi"] = cluster_field(case, seed)
    sk.load_field(lat, st, s["phi"])
    if kind == "flow":
        if case["entry"] == "graph":
            s["graph"] = sk.FlowGraph(lat, st, case["dt"], case["steps"], MODES[case["mode"]])
        elif case["entry"] == "host":
            s["in"] = torch.empty(s["phi"].shape, dtype=s["phi"].dtype, pin_memory=True)
            s["in"].copy_(s["phi"])
            s["out"] = torch.empty(s["phi"].shape, dtype=s["phi"].dtype, pin_memory=True)
            del s["phi"]
    elif kind == "render":
        s["params"] = sk.render_params(case["width"], case["height"], view=render_view(seed),
                                       levelset=case["levelset"], step=case["step"])
        s["work"] = torch.empty(sizes(case) + (4,), dtype=torch.float64, device=DEV)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "batch":
        b = s["batch"]
        for lat, st, phi in zip(b.lats, b.states, s["fields"]):
            sk.load_field(lat, st, phi)
        b.step(case["steps"])
        cur = case["steps"] & 1
        return [(st.phi[cur], st.vel[cur]) for st in b.states]
    lat, st = s["lat"], s["st"]
    if kind == "seed":
        sk.init_field(lat, s["seed"], st)
        return {"phi": st.phi, "vel": st.vel}
    if kind == "energy":
        return sk.energy(lat, st)
    if kind == "observables":
        return sk.observables(lat, st)
    if kind == "render":
        return sk.render(lat, st, s["params"], work=s["work"])
    steps, mode = case["steps"], MODES[case["mode"]]
    if case["entry"] == "host":
        rep = sk.flow_host(lat, case["dt"], steps, mode, st, s["in"], s["out"])
        out = {"phi": s["out"], "vel": st.vel[rep["cur"]]}
    elif case["entry"] == "graph":
        sk.load_field(lat, st, s["phi"])
        s["graph"].launch()
        rep = st.report()
        out = {"phi": st.phi[rep["cur"]], "vel": st.vel[rep["cur"]]}
    else:
        if steps > 1:  # a single step goes on from the state's own field
            sk.load_field(lat, st, s["phi"])
        rep = sk.flow_step(lat, case["dt"], steps, mode, st)
        out = {"phi": st.phi[rep["cur"]], "vel": st.vel[rep["cur"]]}
    out["report"] = {k: rep[k] for k in ("E", "E2", "E4", "E0", "E6", "B", "virial", "delta",
                                         "rms_force", "steps", "arrests")}
    if case["mode"] == "gradient":
        del out["vel"]  # the gradient flow moves no velocity
    return out


def work(case):
    """Bytes: every iteration reads and writes field and velocity once; a loaded
    field is read once.  Operations: the formulas evaluated plainly."""
    if case["kind"] == "batch":
        sides = batch_sides(case, 0)
        inner = sum((N - 4) ** 3 for N in sides)
        total = sum(N ** 3 for N in sides)
        return {"bytes": 16.0 * total + 64.0 * inner * case["steps"],
                "flops": 621.0 * inner * case["steps"]}
    n = sizes(case)
    inner = float((n[0] - 4) * (n[1] - 4) * (n[2] - 4))
    total = float(n[0] * n[1] * n[2])
    site = 32.0 if case["precision"] == 64 else 16.0
    if case["kind"] == "flow":
        per = 888.0 if case["c6"] else 638.0 if case["m_w"] else 621.0
        moved = 2.0 if case["mode"] == "gradient" else 4.0
        load = 0.0 if case["entry"] == "step" and case["steps"] == 1 else site * total
        return {"bytes": load + moved * site * inner * case["steps"],
                "flops": per * inner * case["steps"]}
    if case["kind"] == "energy":
        return {"bytes": site * total, "flops": 190.0 * inner}
    if case["kind"] == "observables":
        return {"bytes": site * total, "flops": 700.0 * inner}
    if case["kind"] == "seed":
        # both field buffers and both velocity buffers
        return {"bytes": 4.0 * site * total, "flops": 150.0 * case["B"] * total}
    pixels = float(case["width"] * case["height"])
    return {"bytes": site * total + 32.0 * total + 16.0 * pixels,
            "flops": 170.0 * total + 20.0 * pixels / case["step"]}


# ------------------------------------------- the same results in 64-bit torch
def d1(a, ax, h):
    """4th-order first derivative along ax; the axis loses two sites per side."""
    s = lambda o: a.narrow(ax, 2 + o, a.shape[ax] - 4)  # noqa: E731
    return (8 * (s(1) - s(-1)) - (s(2) - s(-2))) / (12 * h)


def d2(a, ax, h):
    s = lambda o: a.narrow(ax, 2 + o, a.shape[ax] - 4)  # noqa: E731
    return (16 * (s(1) + s(-1)) - 30 * s(0) - (s(2) + s(-2))) / (12 * h * h)


def inner(a, *axes):
    for ax in axes:
        a = a.narrow(ax, 2, a.shape[ax] - 4)
    return a


def dot(a, b):
    return (a * b).sum(0)


def cross4(a, b, c):
    """eps_ABCD a_B b_C c_D, so that det[p, a, b, c] = p . cross4(a, b, c)."""
    def det3(i, j, k):
        return (a[i] * (b[j] * c[k] - b[k] * c[j]) - a[j] * (b[i] * c[k] - b[k] * c[i])
                + a[k] * (b[i] * c[j] - b[j] * c[i]))
    return torch.stack([det3(1, 2, 3), -det3(0, 2, 3), det3(0, 1, 3), -det3(0, 1, 2)])


def with_boundary(phi):
    """The field as loaded: 64 bits, component first, vacuum on two outer layers."""
    p = torch.zeros((4,) + tuple(phi.shape[:3]), dtype=torch.float64, device=DEV)
    p[0] = 1.0
    p[:, 2:-2, 2:-2, 2:-2] = phi[2:-2, 2:-2, 2:-2].permute(3, 0, 1, 2).double()
    return p


def chunks(n):
    """Ranges of interior x-planes of about 4 M sites."""
    c = max(1, (1 << 22) // (n[1] * n[2]))
    return [(a, min(a + c, n[0] - 4)) for a in range(0, n[0] - 4, c)]


def densities(ph, d, m, m_w=0.0, c6=0.0):
    """{e2, e4, e0, b, e6} summed over the sites, and a_ij."""
    a = [[dot(d[i], d[j]) for j in range(3)] for i in range(3)]
    tr = a[0][0] + a[1][1] + a[2][2]
    sq = sum(a[i][j] ** 2 for i in range(3) for j in range(3))
    u = 1 - ph[0]
    det = dot(ph, cross4(*d))
    sums = torch.stack([tr.sum(), (0.5 * (tr * tr - sq)).sum(),
                        (2 * m * m * u + 0.5 * m_w * m_w * u ** 4).sum(),
                        (-det / (2 * math.pi ** 2)).sum(), (c6 * det * det).sum()])
    return sums, a, tr, det


def energies(sums, h):
    E2, E4, E0, B, E6 = (float(v) * h ** 3 for v in sums)
    return {"E": E2 + E4 + E0 + E6, "E2": E2, "E4": E4, "E0": E0, "B": B,
            "virial": -E2 + E4 - 3 * E0 + 3 * E6, "E6": E6}


def first_derivatives(c, h):
    return [inner(d1(c, 1, h), 2, 3), inner(d1(c, 2, h), 1, 3), inner(d1(c, 3, h), 1, 2)]


def force(c, case):
    """Tangent force on the interior of a haloed chunk, with the density sums."""
    h, m, m_w, c6 = case["h"], case["m"], case.get("m_w", 0.0), case.get("c6", 0.0)
    ph = inner(c, 1, 2, 3)
    fx, fy = d1(c, 1, h), d1(c, 2, h)
    d = [inner(fx, 2, 3), inner(fy, 1, 3), inner(d1(c, 3, h), 1, 2)]
    dd = [[None] * 3 for _ in range(3)]
    dd[0][0] = inner(d2(c, 1, h), 2, 3)
    dd[1][1] = inner(d2(c, 2, h), 1, 3)
    dd[2][2] = inner(d2(c, 3, h), 1, 2)
    dd[0][1] = dd[1][0] = inner(d1(fx, 2, h), 3)
    dd[0][2] = dd[2][0] = inner(d1(fx, 3, h), 2)
    dd[1][2] = dd[2][1] = inner(d1(fy, 3, h), 1)
    sums, a, tr, det = densities(ph, d, m, m_w, c6)
    lap = dd[0][0] + dd[1][1] + dd[2][2]
    br = lap * (1 + tr)
    for i in range(3):
        ci = sum(dot(dd[i][j], d[j]) for j in range(3)) - dot(lap, d[i])
        br = br + d[i] * ci
        for j in range(3):
            br = br - dd[i][j] * a[i][j]
    G = -2 * br
    u = 1 - ph[0]
    G[0] -= 2 * m * m + 2 * m_w * m_w * u ** 3
    if c6:
        P = cross4(*d)
        Q = [-cross4(ph, d[1], d[2]), cross4(ph, d[0], d[2]), -cross4(ph, d[0], d[1])]
        t = 4 * det * P
        for i in range(3):
            t = t - sum(dot(Q[j], dd[i][j]) for j in range(3)) * Q[i]
        G = G + 2 * c6 * t
    return -G + dot(G, ph) * ph, sums


def exact_flow(case, phi):
    """nsteps iterations in 64 bits: field, velocity (site last) and the last report."""
    n, dt, mode = tuple(phi.shape[:3]), case["dt"], case.get("mode", "arrested")
    p = with_boundary(phi)
    v = torch.zeros_like(p)
    before, arrests, rep = math.inf, 0, None
    for _ in range(case["steps"]):
        F = torch.zeros_like(p)
        sums = 0
        for a, b in chunks(n):
            f, s = force(p[:, a:b + 4], case)
            F[:, a + 2:b + 2, 2:-2, 2:-2] = f
            sums = sums + s
        rep = energies(sums, case["h"])
        norm2 = dot(F, F)
        rep["delta"] = math.sqrt(float(norm2.max()))
        rep["rms_force"] = math.sqrt(float(norm2.sum()) / ((n[0] - 4) * (n[1] - 4) * (n[2] - 4)))
        if mode == "gradient":
            t = p + dt * F
        else:
            if mode == "arrested" and rep["E"] > before:
                v.zero_()
                arrests += 1
            before = rep["E"]
            v = v + dt * F
            t = p + dt * v
        del F
        t /= torch.sqrt(dot(t, t))
        i = slice(2, -2)
        p[:, i, i, i] = t[:, i, i, i]
    return p.permute(1, 2, 3, 0), v.permute(1, 2, 3, 0), rep


def exact_observables(case, phi):
    h, m = case["h"], case["m"]
    p = with_boundary(phi)
    n = p.shape[1:]
    ph = inner(p, 1, 2, 3)
    d = first_derivatives(p, h)
    sums, a, tr, det = densities(ph, d, m)
    b = -det / (2 * math.pi ** 2)
    E = energies(sums, h)["E"]
    x = [((torch.arange(2, n[i] - 2, dtype=torch.float64, device=DEV) - 0.5 * (n[i] - 1)) * h)
         .reshape([-1 if k == i else 1 for k in range(3)]) for i in range(3)]
    h3 = h ** 3
    B = h3 * float(b.sum())
    X = [h3 * float((x[i] * b).sum()) / B for i in range(3)]
    r = [x[i] - X[i] for i in range(3)]
    r2 = r[0] ** 2 + r[1] ** 2 + r[2] ** 2
    out = {"B": B, "X": X, "R": math.sqrt(h3 * float((r2 * b).sum()) / B), "E": E}
    out["Q"] = [[h3 * float(((3 * r[i] * r[j] - (r2 if i == j else 0)) * 0.5 * b).sum())
                 for j in range(3)] for i in range(3)]
    t = [d[k] - dot(ph, d[k]) * ph for k in range(3)]
    A = [[dot(t[i], t[j]) for j in range(3)] for i in range(3)]
    trA = A[0][0] + A[1][1] + A[2][2]
    zero = torch.zeros_like(ph[0])
    K = [torch.stack([zero, zero, -ph[3], ph[2]]), torch.stack([zero, ph[3], zero, -ph[1]]),
         torch.stack([zero, -ph[2], ph[1], zero])]
    G = [r[2] * t[1] - r[1] * t[2], r[0] * t[2] - r[2] * t[0], r[1] * t[0] - r[0] * t[1]]

    def inertia(P, Q):
        return [[h3 * float((2 * (dot(P[i], Q[j]) * (1 + trA)
                                  - sum(dot(P[i], t[k]) * dot(Q[j], t[k]) for k in range(3)))).sum())
                 for j in range(3)] for i in range(3)]
    out["U"], out["V"] = inertia(K, K), inertia(G, G)
    out["W"] = [[-v for v in row] for row in inertia(K, G)]
    AA = [[sum(A[i][k] * A[k][j] for k in range(3)) for j in range(3)] for i in range(3)]
    lag = -(trA + 0.5 * (trA * trA - (AA[0][0] + AA[1][1] + AA[2][2])) + 2 * m * m * (1 - ph[0]))
    T = [[2 * A[i][j] * (1 + trA) - 2 * AA[i][j] + (lag if i == j else 0) for j in range(3)]
         for i in range(3)]
    rTr = sum(r[i] * r[j] * T[i][j] for i in range(3) for j in range(3))
    out["D"] = -0.4 * E * h3 * float((rTr - r2 * (T[0][0] + T[1][1] + T[2][2]) / 3).sum())
    return out


def exact_render(case, phi, view):
    p = with_boundary(phi)
    n = p.shape[1:]
    b = torch.zeros(n, dtype=torch.float64, device=DEV)
    i = slice(2, -2)
    b[i, i, i] = -dot(inner(p, 1, 2, 3), cross4(*first_derivatives(p, case["h"]))) / (2 * math.pi ** 2)
    b = b / b.max()
    pion = torch.sqrt(p[1] ** 2 + p[2] ** 2 + p[3] ** 2)
    unit = [torch.where(pion > 0, p[k] / torch.where(pion > 0, pion, 1.0), 0.0) for k in (1, 2, 3)]
    vol = torch.stack([b] + unit, -1).reshape(-1, 4)
    W, H, step = case["width"], case["height"], case["step"]
    half = [0.5 * (k - 1) for k in n]
    s = max(half)
    f64 = dict(dtype=torch.float64, device=DEV)
    u = ((2 * (torch.arange(W, **f64) + 0.5) / W - 1) * (W / H)).repeat(H)
    v = (2 * (torch.arange(H, **f64) + 0.5) / H - 1).repeat_interleave(W)
    ray = torch.stack([u, v, torch.full_like(u, -2.0)])
    ray = ray / torch.sqrt((ray * ray).sum(0))
    R = torch.tensor(view, **f64)
    d = torch.stack([R[k, 0] * ray[0] + R[k, 1] * ray[1] + R[k, 2] * ray[2] for k in range(3)])
    o = [float(R[k, 2]) * 4.0 for k in range(3)]
    near, far = torch.zeros_like(u), torch.full_like(u, 1e300)
    for k in range(3):
        lim = half[k] / s
        t0, t1 = (-lim - o[k]) / d[k], (lim - o[k]) / d[k]
        near = torch.maximum(near, torch.minimum(t0, t1))
        far = torch.minimum(far, torch.maximum(t0, t1))
    out = torch.zeros((4, W * H), **f64)
    t = near.clone()
    alive = torch.nonzero(t <= far).flatten()
    while alive.numel():
        ta = t[alive]
        g = [(o[k] + ta * d[k][alive]) * s + half[k] for k in range(3)]
        g = [x.clamp(0, n[k] - 1) for k, x in enumerate(g)]
        c = [torch.clamp(x.floor().long(), max=n[k] - 2) for k, x in enumerate(g)]
        w = [x - y for x, y in zip(g, c)]
        smp = 0
        for q in range(8):
            e = [q & 1, (q >> 1) & 1, (q >> 2) & 1]
            wt = 1
            for k in range(3):
                wt = wt * (w[k] if e[k] else 1 - w[k])
            smp = smp + wt[:, None] * vol[((c[0] + e[0]) * n[1] + c[1] + e[1]) * n[2] + c[2] + e[2]]
        inp = (smp[:, 0] - case["levelset"]) * 4.0
        col = torch.stack([inp * inp * smp[:, 1], inp * inp * smp[:, 2], inp * inp * smp[:, 3], inp])
        cur = out[:, alive]
        out[:, alive] = torch.where(inp >= 0, cur + col * (1 - cur[3]), cur)
        t[alive] = ta + step
        alive = alive[(t[alive] <= far[alive]) & (out[3, alive] <= 0.95)]
    return out.clamp(0, 1).T.reshape(H, W, 4)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        got = []
        for k, N in enumerate(batch_sides(case, seed)):
            p, v, _ = exact_flow(case, noise_field(case, N, 1000 * seed + k))
            got.append((p, v))
        return got
    n = sizes(case)
    if kind == "seed":
        pos, quat = constituents(case, seed)
        phi = torch.zeros(n + (4,), dtype=torch.float64, device=DEV)
        phi[..., 0] = 1.0
        i = slice(2, -2)
        for a, b in chunks(n):
            phi[a + 2:b + 2, i, i] = product_field(n, case["h"], pos, quat, torch.float64, 1.0,
                                                   case["symmetrise"], a + 2, b + 2)[:, i, i]
        return {"phi": torch.stack([phi, phi]), "vel": None}
    phi = cluster_field(case, seed)
    if kind == "flow":
        p, v, rep = exact_flow(case, phi)
        out = {"phi": p, "vel": v, "report": rep}
        if case["mode"] == "gradient":
            del out["vel"]
        return out
    if kind == "energy":
        p, sums = with_boundary(phi), 0
        for a, b in chunks(n):
            c = p[:, a:b + 4]
            sums = sums + densities(inner(c, 1, 2, 3), first_derivatives(c, case["h"]), case["m"])[0]
        out = energies(sums, case["h"])
        del out["E6"]
        return out
    if kind == "observables":
        return exact_observables(case, phi)
    return exact_render(case, phi, render_view(seed))
