"""The work that a user of this framework has it do, as cases that can be timed.

Every case is a whole call or a whole hot path through the public entry points
(``lbm_em.Solver``, ``lbm_em.run_instance``, ``lbm_em.Batch``, ``trajectory.janus_map``), on
the workloads of ``workloads.py`` and the maps of ``trajectory.py`` or on problems of the same
families at other sizes.  The kinds:

* ``call``    ``run_instance``: create a solver, march, accumulate a period, integrate, destroy.
* ``maps``    a solver created from host permittivity and conductor maps, marched, read back
              (forces, phasors, the three fields) and destroyed.
* ``solver``  a solver that the program keeps: next geometry, reset, march, accumulate, integrate,
              read the contour's phasors.
* ``march``   a solver in mid-run that goes on for some periods and reports the force of the last.
* ``grid``    ``trajectory.janus_map``: a force and torque map over materials and orientations.
* ``design``  a batch of uneven instances that the program keeps and runs again.
"""
import math
import random

import numpy as np
import torch

from paper_2509_22308_gb300 import lbm_em as L
from paper_2509_22308_gb300 import trajectory as TR

# Arithmetic operations of one site update: the moments (D 5, E/3 1, H_x and H_y 5 each), the
# thirds of H (2), the sums of the equilibria (4) and the 11 relaxed populations.
OPS = 33
POPULATIONS = 11
SITE_BYTES = {"f64": 88, "f32": 44, "f16dev": 34, "f32x2": 88}
EXACT_UPDATES = 30e9  # site updates that the reference below does in well under 20 s


def listed():
    return [
        # One small scattering problem from start to end: the smoke check's instance.
        dict(name="call_67x45_f64", kind="call", form="f64", nx=67, ny=45, a=9.0, R=14.0, period=36, periods=4,
             body="md"),
        # A scatterer given as maps (graded permittivity, conducting pieces), TE, read back whole.
        dict(name="maps_384x300_f32_te", kind="maps", form="f32", te=True, nx=384, ny=300, a=40.0, R=66.0, period=90,
             periods=12, body="graded"),
        # The paper's plain method on the homogeneous cylinder (workloads.homogeneous_dielectric_256).
        dict(name="homog_256_f64", kind="solver", form="f64", nx=256, ny=256, a=20.0, R=40.0, period=120, periods=20,
             body="homog"),
        # The benchmark's instance (workloads.md_janus_512) in the forms a user chooses between.
        dict(name="md_512_f64", kind="solver", form="f64", nx=512, ny=512, a=32.0, R=64.0, period=96, periods=30,
             body="md"),
        dict(name="md_512_f32", kind="solver", form="f32", nx=512, ny=512, a=32.0, R=64.0, period=96, periods=30,
             body="md"),
        dict(name="md_512_f32x2", kind="solver", form="f32x2", nx=512, ny=512, a=32.0, R=64.0, period=96, periods=30,
             body="md"),
        # A large cylinder until its forces have settled (workloads.dielectric_janus_2048, k0 a = 20).
        dict(name="dj_2048_f32", kind="solver", form="f32", nx=2048, ny=2048, a=128.0, R=204.8, period=120,
             periods=45, body="dj"),
        # The same with the compact storage, going on from a developed field.
        dict(name="dj_2048_f16dev", kind="march", form="f16dev", nx=2048, ny=2048, a=128.0, R=204.8, period=120,
             before=3840, periods=8, body="dj"),
        # The paper's metallo-dielectric map (Sec. IV.A: 160^2, a = 40, 30 periods), part of it.
        dict(name="grid_md_160", kind="grid", form="f32", a=40, L_over_a=4, periods=30, conv=0.0, n_eps=5, n_phi=36,
             body="md"),
        # The paper's dielectric map (Sec. IV.B: 200^2, a = 50), each instance until it has settled.
        dict(name="grid_dj_200_conv", kind="grid", form="f32", a=50, L_over_a=4, periods=40, conv=1e-3, n_eps=4,
             n_phi=24, body="dj"),
        # A design diagram over uneven lattices (workloads.design_map_256), a fifth of it.
        dict(name="design_48_f32", kind="design", form="f32", n=48, sizes="16,32,64", periods=20, body="dj"),
        # The large single domain (workloads.md_janus_8192), the cylinder near the source side so that
        # the field around it has developed.
        dict(name="md_8192_f32", kind="march", form="f32", nx=8192, ny=8192, a=512.0, R=768.0, cx=1000.0, period=240,
             before=5520, periods=4, body="md"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["call", "maps", "solver", "solver", "solver", "solver", "march", "grid", "grid", "design"])
    if kind == "design":
        return dict(kind=kind, form=rng.choice(["f32", "f32", "f32x2"]), n=rng.randint(8, 40),
                    sizes=rng.choice(["16,32", "16,32,64", "12,20,33"]), periods=rng.randint(12, 20), body="dj")
    if kind == "grid":
        a = rng.randint(16, 50)
        n_eps, n_phi = rng.randint(2, 6), rng.randint(8, 36)
        return dict(kind=kind, form="f32", a=a, L_over_a=rng.choice([4, 5]), periods=rng.randint(14, 30),
                    conv=rng.choice([0.0, 0.0, 1e-3]), n_eps=n_eps, n_phi=n_phi, body=rng.choice(["md", "dj"]))
    form = rng.choice(["f32", "f32", "f32", "f64", "f16dev", "f32x2"])
    te = form != "f16dev" and rng.random() < 0.25
    if kind == "march":  # large lattices: the field around the body is developed before
        form = rng.choice(["f32", "f16dev"])
        nx, ny = _logint(rng, 900, 6000), _logint(rng, 900, 6000)
        a = float(rng.randint(40, 120))
        return dict(kind=kind, form=form, te=form == "f32" and rng.random() < 0.25, nx=nx, ny=ny, a=a, R=1.6 * a,
                    cx=float(rng.randint(220, 400)), period=rng.randint(60, 160),
                    before=rng.randint(1800, 2600), periods=rng.randint(2, 6), body=rng.choice(["md", "dj"]))
    top = {"f64": 640, "f32x2": 768, "f32": 1800, "f16dev": 1800}[form]
    if kind == "call":
        top = min(top, 320)
    if kind == "maps":
        top = min(top, 640)
    n = _logint(rng, 48, top)
    nx, ny = max(48, int(n * rng.uniform(0.8, 1.25))), max(48, int(n * rng.uniform(0.8, 1.25)))
    a = round(min(nx, ny) * rng.uniform(0.06, 0.16), 2)
    R = round(a * rng.uniform(1.4, 2.0) + 2.0, 2)
    period = rng.randint(30, 150)
    periods = int(math.ceil(1.5 * (nx + 2 * R) / period)) + rng.randint(2, 6)
    c = dict(kind=kind, form=form, te=te, nx=nx, ny=ny, a=a, R=R, period=period, periods=periods,
             body="graded" if kind == "maps" else rng.choice(["md", "dj", "homog"]))
    if kind == "solver":
        c["source"] = rng.choice(["hard", "hard", "open"])
    return c


# ---- inputs ---------------------------------------------------------------------------------

def _body(case, rng):
    """(phi0, eps1, eps2, pec2) of one Janus cylinder of the case's family."""
    phi0 = rng.uniform(0.0, math.pi)
    if case["body"] == "homog":
        e = rng.uniform(2.0, 4.0)
        return phi0, e, e, False
    if case["body"] == "md":
        return phi0, rng.uniform(2.0, 10.0), 1.0, True
    return phi0, 2.0, rng.uniform(2.0, 12.0), False


def _graded(case, seed):
    """A graded-index disc in 24 steps with an off-centre conducting inclusion: (eps, pec) maps."""
    rng = random.Random(seed)
    nx, ny, a = case["nx"], case["ny"], case["a"]
    peak, phi, off = rng.uniform(2.0, 6.0), rng.uniform(0.0, 2.0 * math.pi), rng.uniform(0.2, 0.5) * a
    x, y = np.arange(nx)[None, :] - (nx - 1) / 2.0, np.arange(ny)[:, None] - (ny - 1) / 2.0
    r = np.sqrt(x * x + y * y) / a
    eps = np.where(r <= 1.0, 1.0 + (peak - 1.0) * np.ceil(24.0 * np.maximum(0.0, 1.0 - r * r)) / 24.0, 1.0)
    pec = ((x - off * math.cos(phi)) ** 2 + (y - off * math.sin(phi)) ** 2 <= (0.2 * a) ** 2).astype(np.uint8)
    return eps, pec


def _instance(case, seed):
    phi0, e1, e2, pec = _body(case, random.Random(seed))
    return dict(nx=case["nx"], ny=case["ny"], a=case["a"], phi0=phi0, eps1=e1, eps2=e2, pec2=pec, R=case["R"],
                period=case["period"], periods=case.get("periods", 1), ramp=case["period"])


def _design(case, seed):
    """Instances as workloads.design_map_256 draws them, from the given radii."""
    rng = random.Random(seed)
    sizes = [int(v) for v in case["sizes"].split(",")]
    out = []
    for i in range(case["n"]):
        a = sizes[i % len(sizes)]
        out.append(dict(nx=16 * a, ny=16 * a, a=float(a), phi0=rng.uniform(0.0, math.pi), eps1=2.0,
                        eps2=rng.uniform(2.0, 12.0), pec2=False, period=3 * a, periods=case["periods"], R=1.6 * a,
                        ramp=3 * a))
    rng.shuffle(out)
    return out


def _grid(case, seed):
    """Materials and orientations of a map."""
    rng = random.Random(seed)
    e = sorted(rng.uniform(1.5, 5.0) for _ in range(case["n_eps"]))
    phi0 = rng.uniform(0.0, 0.1)
    return ([(v, 1.0, True) if case["body"] == "md" else (2.0, v, False) for v in e],
            [phi0 + 2.0 * math.pi * k / case["n_phi"] for k in range(case["n_phi"])])


def _pol(case):
    return "te" if case.get("te") else "tm"


def prepare(case, seed):
    s = dict(case=case)
    kind = case["kind"]
    if kind == "grid":
        s["materials"], s["phi0"] = _grid(case, seed)
        return s
    if kind == "design":
        s["batch"] = L.Batch(_design(case, seed), case["form"])
        return s
    if kind == "maps":
        s["eps"], s["pec"] = _graded(case, seed)
        return s
    inst = s["inst"] = _instance(case, seed)
    if kind == "call":
        return s
    src = L.make_source(case["period"], kind=L.SRC_OPEN if case.get("source") == "open" else L.SRC_HARD)
    s["janus"] = L.make_janus(inst["a"], inst["phi0"], inst["eps1"], inst["eps2"], inst["pec2"], cx=case.get("cx"))
    s["contour"] = L.make_contour(inst["R"], inst["a"], cx=case.get("cx"))
    s["solver"] = L.Solver(case["nx"], case["ny"], case["form"], janus=s["janus"], source=src, polarization=_pol(case))
    if kind == "march":
        s["solver"].step(case["before"])
        s["solver"].sync()
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "call":
        return {"force": L.run_instance(state["inst"], case["form"], polarization=_pol(case))}
    if kind == "grid":
        F, steps = TR.janus_map(state["materials"], state["phi0"], a=case["a"], L_over_a=case["L_over_a"],
                                periods=case["periods"], precision=case["form"], conv_tol=case["conv"])
        return {"force": F, "steps": steps}
    if kind == "design":
        state["batch"].run()
        F, status = state["batch"].results()
        return {"force": F, "status": status}
    T = case["period"]
    if kind == "maps":
        with L.Solver(case["nx"], case["ny"], case["form"], eps_map=state["eps"], pec_mask=state["pec"],
                      source=L.make_source(T), polarization=_pol(case)) as s:
            s.step((case["periods"] - 1) * T)
            F = s.force_torque(L.make_contour(case["R"], case["a"]))
            return {"force": F, "phasors": s.phasors()[1], "fields": s.fields()}
    s = state["solver"]
    if kind == "solver":
        s.set_janus(state["janus"])
        s.reset()
    s.step((case["periods"] - 1) * T)
    F = s.force_torque(state["contour"])
    return {"force": F, "phasors": s.phasors()[1]}


# ---- what a pass cannot do without ----------------------------------------------------------

def _updates(case):
    """(site updates, sites) of one pass."""
    if case["kind"] == "grid":  # with convergence exits at most this
        n = int(round(case["L_over_a"] * case["a"]))
        sites = case["n_eps"] * case["n_phi"] * n * n
        return sites * case["periods"] * 3 * case["a"], sites
    if case["kind"] == "design":
        sizes = [int(v) for v in case["sizes"].split(",")]
        a = [sizes[i % len(sizes)] for i in range(case["n"])]
        return sum((16 * v) ** 2 * 3 * v * case["periods"] for v in a), sum((16 * v) ** 2 for v in a)
    sites = case["nx"] * case["ny"]
    return sites * case["periods"] * case["period"], sites


def work(case):
    """The operations of every site update; the state once read and once written, and the ids."""
    up, sites = _updates(case)
    return {"bytes": float(sites * (2 * SITE_BYTES[case["form"]] + 1)), "flops": float(up * OPS)}


# ---- the same in 64 bits --------------------------------------------------------------------
# The D3Q7 scheme of arXiv 2509.22308, Sec. III, for b lattices at once: populations
# [b, ny, nx] of the in-plane components that the triple (TM: E_z, H_x, H_y) can reach.

class _Reference:
    def __init__(self, eps, pec, T, ramp, te, source):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.eps = torch.as_tensor(eps, dtype=torch.float64, device=dev)
        free = ~torch.as_tensor(pec, dtype=torch.bool, device=dev)
        self.inv = torch.where(free, 1.0 / self.eps, 0.0)
        # weight of the z pair in D with the rest population folded in (none of either in a conductor)
        self.wz = torch.where(free, 6.0 * self.eps - 4.0, 0.0)
        self.T, self.ramp, self.te, self.open, self.t = T, ramp, te, source == "open", 0
        self.p = {k: torch.zeros_like(self.eps) for k in "z e w n s xe xw xz yn ys yz".split()}
        zt = np.exp(-2j * math.pi / T)
        self.w = (3.0 - zt) / (zt * (3.0 * zt - 1.0))
        self.P = 2j / (3.0 * (self.w * zt + 1.0))

    def pulled(self):
        """Populations of the current time before the collision: streamed, with the open edges
        (zero gradient) and the source."""
        p, q = self.p, {}
        for k, (d, back) in dict(e=(2, False), xe=(2, False), w=(2, True), xw=(2, True), n=(1, False), yn=(1, False),
                                 s=(1, True), ys=(1, True)).items():
            m = p[k].shape[d]
            edge = p[k].narrow(d, m - 1 if back else 0, 1)
            q[k] = torch.cat([p[k].narrow(d, 1, m - 1), edge] if back else [edge, p[k].narrow(d, 0, m - 1)], d)
        q["z"], q["xz"], q["yz"] = p["z"], p["xz"], p["yz"]
        t = self.t
        if t >= 1:
            f = math.sin(0.5 * math.pi * t / self.ramp) ** 2 if t < self.ramp else 1.0
            zt = np.exp(-2j * math.pi * (t % self.T) / self.T)
            inc, ahead = f * (self.P * zt).real, f * (self.P * self.w * zt).real
            if self.open:
                q["e"][:, :, 0] += inc - ahead
            else:
                q["e"][:, :, 0] = inc
                q["xe"][:, :, 0] = 0.0
        return q

    def triple(self, q):
        D = self.wz * q["z"] + (q["e"] + q["w"] + q["n"] + q["s"])
        if not self.te:
            return (D * self.inv, 2.0 * q["xz"] + q["xe"] + q["xw"] + q["n"] - q["s"],
                    2.0 * q["yz"] + q["yn"] + q["ys"] + q["w"] - q["e"])
        Dx = self.wz * q["xz"] + (q["xe"] + q["xw"] + q["yn"] + q["ys"])
        return 2.0 * q["yz"] + q["e"] - q["w"] + q["ys"] - q["yn"], Dx * self.inv, D * self.inv

    def energy(self, f):
        E2 = f[1] ** 2 + f[2] ** 2 if self.te else f[0] ** 2
        H2 = f[0] ** 2 if self.te else f[1] ** 2 + f[2] ** 2
        return (0.5 * (self.eps * E2 + H2)).sum((1, 2))

    def step(self):
        """One step; returns the triple before the collision."""
        q = self.pulled()
        f = self.triple(q)
        a, b, c = (v / 3.0 for v in f)
        eq = (dict(z=a, e=a - c, w=a + c, n=a + b, s=a - b, xe=b, xw=b, xz=b, yn=c, ys=c, yz=c) if not self.te else
              dict(z=c, e=c + a, w=c - a, n=c, s=c, xe=b, xw=b, xz=b, yn=b - a, ys=b + a, yz=a))
        self.p = {k: eq[k] - q[k] for k in q}
        self.t += 1
        return f


def _contour(nx, ny, cx, cy, R):
    """Points of the contour, their four sites and weights; the sites in order of first use."""
    n = int(2 * math.ceil(2.0 * math.pi * R))
    phi = 2.0 * math.pi * np.arange(n) / n
    px, py = cx + R * np.cos(phi), cy + R * np.sin(phi)
    i, j = np.floor(px).astype(int), np.floor(py).astype(int)
    fx, fy = px - i, py - j
    xs, ys = np.stack([i, i + 1, i, i + 1], 1), np.stack([j, j, j + 1, j + 1], 1)
    w = np.stack([(1 - fx) * (1 - fy), fx * (1 - fy), (1 - fx) * fy, fx * fy], 1)
    key = (ys * nx + xs).reshape(-1)
    _, first = np.unique(key, return_index=True)
    order = key[np.sort(first)]
    at = {k: m for m, k in enumerate(order)}
    return dict(n=n, phi=phi, R=R, w=w, site=np.array([at[k] for k in key]).reshape(n, 4), x=order % nx, y=order // nx)


def _force(c, ph, a):
    """Period-averaged Maxwell stress over the contour (Sec. II.B) from [sites, 6] phasors."""
    v = (c["w"][:, :, None] * ph[c["site"]]).sum(1)
    f = [v[:, 2 * k] + 1j * v[:, 2 * k + 1] for k in range(3)]
    half = 0.5 * sum(abs(x) ** 2 for x in f)
    xx, yy = 0.5 * (abs(f[1]) ** 2 - half), 0.5 * (abs(f[2]) ** 2 - half)
    xy = 0.5 * (f[1] * np.conj(f[2])).real
    nx, ny = np.cos(c["phi"]), np.sin(c["phi"])
    tx, ty = xx * nx + xy * ny, xy * nx + yy * ny
    dl, F0 = 2.0 * math.pi * c["R"] / c["n"], math.pi * a / 4.0
    return np.array([tx.sum() * dl / F0, ty.sum() * dl / F0, (c["R"] * (nx * ty - ny * tx)).sum() * dl / (2 * F0 * a)])


def _janus_maps(insts, cx=None):
    eps, pec = [], []
    for i in insts:
        x = np.arange(i["nx"])[None, :] - ((i["nx"] - 1) / 2.0 if cx is None else cx)
        y = np.arange(i["ny"])[:, None] - (i["ny"] - 1) / 2.0
        inside = x * x + y * y <= i["a"] * i["a"]
        two = x * -math.sin(i["phi0"]) + y * -math.cos(i["phi0"]) > 1e-9
        eps.append(np.where(inside & two, i["eps1"], np.where(inside & ~two & (not i["pec2"]), i["eps2"], 1.0)))
        pec.append(inside & ~two & i["pec2"])
    return np.stack(eps), np.stack(pec)


def _solve(ref, c, before, T, conv=0.0, least=1, limit=None):
    """Marches ``before`` steps and accumulates the next T: (phasors [b, sites, 6], steps [b]).  With
    ``conv`` each lattice stops as the batch's convergence exits do."""
    b, dev = ref.eps.shape[0], ref.eps.device
    x, y = torch.as_tensor(c["x"], device=dev), torch.as_tensor(c["y"], device=dev)
    acc = torch.zeros(b, len(c["x"]), 6, dtype=torch.float64, device=dev)
    start = torch.full((b,), before, device=dev)
    prev, settled, last = [-1.0] * b, [0] * b, before + T
    t0 = ref.t
    while ref.t - t0 < last:
        t = ref.t - t0
        f = ref.step()
        if conv > 0.0 and t > 0 and t % T == 0:
            W = ref.energy(f).tolist()
            for k in range(b):
                if t >= int(start[k]):
                    continue
                settled[k] = settled[k] + 1 if prev[k] > 0.0 and abs(W[k] - prev[k]) <= conv * W[k] else 0
                prev[k] = W[k]
                if settled[k] >= 2 and t // T + 1 >= least:
                    start[k] = t + 1
            last = int(start.max()) + T
        if conv > 0.0 or t >= before:
            on = ((t >= start) & (t < start + T)).to(torch.float64)[:, None, None]
            ph = 2.0 * math.pi * ((t + t0) % T) / T
            v = torch.stack([g[:, y, x] for g in f], 2)
            acc += on * torch.stack([v * math.cos(ph), v * math.sin(ph)], 3).reshape(b, -1, 6)
    return (acc * (2.0 / T)).cpu().numpy(), (start + T).cpu().numpy()


def exact(case, seed):
    if _updates(case)[0] + case.get("before", 0) * case.get("nx", 0) * case.get("ny", 0) > EXACT_UPDATES:
        return None
    te, kind, T = bool(case.get("te")), case["kind"], case.get("period")
    if kind == "grid":
        a, n = float(case["a"]), int(round(case["L_over_a"] * case["a"]))
        materials, phi = _grid(case, seed)
        T = int(round(3 * a))
        insts = [dict(nx=n, ny=n, a=a, phi0=p, eps1=m[0], eps2=m[1], pec2=m[2]) for m in materials for p in phi]
        ref = _Reference(*_janus_maps(insts), T, T, te, "hard")
        c = _contour(n, n, (n - 1) / 2.0, (n - 1) / 2.0, 1.5 * a)
        ph, steps = _solve(ref, c, (case["periods"] - 1) * T, T, case["conv"], min(8, case["periods"]))
        shape = (len(materials), len(phi))
        return {"force": np.stack([_force(c, v, a) for v in ph]).reshape(shape + (3,)), "steps": None}
    if kind == "design":
        insts, F = _design(case, seed), {}
        for a in sorted({i["a"] for i in insts}):
            at = [k for k, i in enumerate(insts) if i["a"] == a]
            n, T = insts[at[0]]["nx"], insts[at[0]]["period"]
            ref = _Reference(*_janus_maps([insts[k] for k in at]), T, T, te, "hard")
            c = _contour(n, n, (n - 1) / 2.0, (n - 1) / 2.0, insts[at[0]]["R"])
            ph, _ = _solve(ref, c, (case["periods"] - 1) * T, T)
            F.update({k: _force(c, v, a) for k, v in zip(at, ph)})
        return {"force": np.stack([F[k] for k in range(len(insts))]), "status": None}
    if kind == "maps":
        eps, pec = _graded(case, seed)
        eps, pec = eps[None], pec[None]
    else:
        eps, pec = _janus_maps([_instance(case, seed)], case.get("cx"))
    ref = _Reference(eps, pec, T, T, te, case.get("source", "hard"))
    nx, ny = case["nx"], case["ny"]
    c = _contour(nx, ny, case.get("cx", (nx - 1) / 2.0), (ny - 1) / 2.0, case["R"])
    ph, _ = _solve(ref, c, case.get("before", 0) + (case["periods"] - 1) * T, T)
    out = {"force": _force(c, ph[0], case["a"])}
    if kind != "call":
        out["phasors"] = ph[0]
    if kind == "maps":
        out["fields"] = tuple(v[0].cpu().numpy() for v in ref.triple(ref.pulled()))
    return out
