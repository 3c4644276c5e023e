"""The work that is measured: whole calls of the coupled LBM-DEM step, its fluid
step alone, a batch of boxes and the linked-cell sort, each through the Python
entry points of the package, over the sizes, forms and closures they are used at.

Every coupled case is a user's loop body: advance the box by a few steps, then
read the particles and the fluid velocity back.  `exact` is an independent
64-bit restatement of the method in plain torch tensor operations.
"""
import math

import numpy as np
import torch

from paper_1711_00336_gb300 import dps

DEV = "cuda" if torch.cuda.is_available() else "cpu"
PI = math.pi

# ---- the cases -------------------------------------------------------------------
# kind "coupled": box nx x ny x nz, px/py/pz periodic (1) or walls (0), `form` the
# precision form, `eps` solid volume fraction (0: one sphere), d the sphere diameter,
# `poly` the relative spread of the diameters, `touch` the spacing lost to overlap
# (contacts of a developed suspension), `steps` coupled steps per pass.
COUPLED = dict(kind="coupled", form="f64", nx=64, ny=64, nz=64, px=1, py=1, pz=1, tau=0.55, eps=0.2, d=1.5,
               poly=0.0, touch=0.0, h_c=1.5, T_c=0.5, e_n=0.88, n_int=2, n_dem=10, fb_mode=1, Re=0.1, lift=0,
               eilers=0, smag=0, steps=2)


def _coupled(**kw):
    return {**COUPLED, **kw}


def listed():
    return [
        # one settling sphere between walls (the method's validation run, thousands of steps): every
        # launch is small, so latency is all there is
        _coupled(name="sphere_f64", nx=32, ny=32, nz=64, pz=0, tau=0.65, eps=0.0, d=0.8, h_c=1.0, T_c=1.0,
                 e_n=0.9, n_int=1, fb_mode=0, steps=20),
        # a wall-bounded suspension of 5000 spheres, the second line of the benchmark
        _coupled(name="walls_f64", pz=0, tau=0.65, eps=0.01, d=1.0, h_c=1.0, T_c=1.0, e_n=0.9, n_int=1, fb_mode=0,
                 Re=0.02, steps=10),
        # the benchmark's workload: the largest single box, 1.9 million spheres, plain FP64 method
        _coupled(name="settling_f64_256", nx=256, ny=256, nz=256, steps=2),
        # a dense, developed suspension (pairs in contact), ragged box, FP64
        _coupled(name="dense_f64_ragged", nx=101, ny=90, nz=77, eps=0.36, d=1.25, touch=0.006, h_c=1.25,
                 n_int=4, n_dem=5, steps=4),
        # all closures on (lift, Eilers, Smagorinsky), walls on two axes, odd sizes, FP64
        _coupled(name="closures_f64_walls", nx=75, ny=61, nz=90, py=0, pz=0, tau=0.6, eps=0.1, d=1.0, h_c=0.5,
                 fb_mode=0, Re=0.02, lift=1, eilers=1, smag=1, steps=4),
        # production form FP32 on a dense box
        _coupled(name="settling_f32_dense", form="f32", nx=192, ny=192, nz=192, eps=0.38, steps=2),
        # FP16 storage on a large dilute box: the fluid side dominates
        _coupled(name="settling_f16s_dilute", form="f16s", nx=256, ny=256, nz=256, eps=0.05, steps=4),
        # hindered settling at the subcycle counts of the paper (10 x 50 substeps a step), small box, FP32
        _coupled(name="hindered_f32_32", form="f32", nx=32, ny=32, nz=32, tau=0.5045, eps=0.3, d=1.0, h_c=1.0,
                 n_int=10, n_dem=50, Re=0.5, lift=1, eilers=1, smag=1, steps=1),
        # the fluid step alone (fluid-only use), FP64 and the FP16-storage form at an odd row length
        dict(name="fluid_f64", kind="fluid", form="f64", nx=128, ny=128, nz=128, px=1, py=1, pz=0, tau=0.6, steps=60),
        dict(name="fluid_f16s_odd", kind="fluid", form="f16s", nx=161, ny=150, nz=139, px=1, py=0, pz=1, tau=0.7,
             steps=200),
        # many uneven boxes advanced by one launch per phase (parameter studies, the server's inner loop)
        dict(name="batch_f32", kind="batch", form="f32", boxes=12, lo=24, hi=80, eps_lo=0.02, eps_hi=0.35, d=1.3,
             steps=4),
        # the linked-cell sort op on device buffers
        dict(name="cell_sort", kind="sort", nx=160, ny=150, nz=141, px=1, py=1, pz=0, np=1000003),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["coupled"] * 5 + ["fluid"] * 2 + ["batch", "sort"])
    form = rng.choice(["f64", "f64", "f32", "f16s"])
    n = [max(20, int(round(_log(rng, 24, 150) * rng.uniform(0.8, 1.25)))) for _ in range(3)]
    per = [int(rng.random() < 0.75) for _ in range(3)]
    if kind == "sort":
        return dict(kind="sort", nx=n[0], ny=n[1], nz=n[2], px=per[0], py=per[1], pz=per[2],
                    np=int(_log(rng, 1000, 2e6)))
    if kind == "batch":
        return dict(kind="batch", form=rng.choice(["f32", "f64", "f16s"]), boxes=rng.randint(3, 14), lo=24,
                    hi=rng.randint(32, 72), eps_lo=0.02, eps_hi=rng.uniform(0.1, 0.35), d=rng.uniform(1.2, 1.5),
                    steps=4)
    if kind == "fluid":
        return dict(kind="fluid", form=form, nx=n[0], ny=n[1], nz=n[2], px=per[0], py=per[1], pz=per[2],
                    tau=rng.uniform(0.55, 0.9), steps=rng.randint(20, 60) * (1 if form == "f64" else 3))
    dense = rng.random() < 0.4
    walls = not all(per)
    d = rng.uniform(1.2, 1.5) if dense else rng.uniform(0.9, 1.5)
    return _coupled(form=form, nx=n[0], ny=n[1], nz=n[2], px=per[0], py=per[1], pz=per[2],
                    tau=0.55 if not walls else 0.6, eps=rng.uniform(0.25, 0.36) if dense else _log(rng, 0.01, 0.2),
                    d=d, poly=rng.choice([0.0, 0.04]), touch=rng.choice([0.0, 0.004]),
                    h_c=rng.choice([0.5, 1.0, 1.5]), n_int=4 if dense else 2, n_dem=5 if dense else 10,
                    fb_mode=0 if walls else 1, Re=0.02 if walls else 0.1, lift=int(rng.random() < 0.3),
                    eilers=int(rng.random() < 0.3), smag=int(rng.random() < 0.3), steps=rng.randint(2, 4))


# ---- inputs ------------------------------------------------------------------------
def _spheres(n, per, eps, d, poly, touch, rng):
    """Spheres on a random subset of a jittered cubic lattice (all but `touch` of
    the spare spacing is used, so lattice neighbours come close to contact, or
    overlap by up to 2 `touch`); wall axes keep the spheres off the faces."""
    L = [n[a] if per[a] else n[a] - 0.1 for a in range(3)]
    off = [0.0 if per[a] else 0.05 for a in range(3)]
    dmax = d * (1.0 + poly)
    m = [max(1, int(L[a] / (1.02 * dmax))) for a in range(3)]
    count = 1 if eps <= 0 else max(1, int(round(eps * n[0] * n[1] * n[2] / (PI / 6 * d ** 3))))
    sites = m[0] * m[1] * m[2]
    count = min(count, sites)
    if eps <= 0:
        x = np.array([[n[0] / 2, n[1] / 2, 0.75 * n[2]]]) + rng.uniform(-0.5, 0.5, (1, 3))
    else:
        s = rng.permutation(sites)[:count] if count * 4 > sites else rng.choice(sites, count, replace=False)
        ijk = np.stack([s % m[0], (s // m[0]) % m[1], s // (m[0] * m[1])], 1).astype(float)
        a = np.array([L[k] / m[k] for k in range(3)])
        jit = np.maximum((a - dmax) / 2 * 0.999, 0.0)
        r = rng.uniform(-1.0, 1.0, (count, 3))
        x = (ijk + 0.5) * a + r * jit + np.array(off)
        for k in range(3):
            if per[k]:
                x[:, k] = np.mod(x[:, k] + touch * np.sign(r[:, k]), n[k])
    dia = d * (1.0 + poly * rng.uniform(-1.0, 1.0, len(x)))
    u = 1e-3 * rng.standard_normal((len(x), 3))
    w = 1e-3 * rng.standard_normal((len(x), 3))
    return dict(x=x, u=u, w=w, d=dia, rho_p=np.full(len(x), 2.5))


def _closure(c):
    nu = (c["tau"] - 0.5) / 3.0
    g = 18.0 * nu * (c["Re"] * nu / c["d"]) / (1.5 * c["d"] ** 2)
    return dict(g=(0.0, 0.0, -g), fb_mode=c["fb_mode"], fb=(0.0, 0.0, 0.0), e_n=c["e_n"], mu_c=0.25, T_c=c["T_c"],
                h_c=c["h_c"], h_min=1e-5, C_am=0.5, n_int=c["n_int"], n_dem=c["n_dem"], lub_limiter=1, lub_cap=0.25,
                eps_min=0.05, skin=0.5, lift=c["lift"], eilers=c["eilers"], smagorinsky=c["smag"])


def _geometry(c):
    return (c["nx"], c["ny"], c["nz"]), (c["px"], c["py"], c["pz"])


def _coupled_inputs(c, seed):
    n, per = _geometry(c)
    return _spheres(n, per, c["eps"], c["d"], c["poly"], c["touch"], np.random.default_rng(seed))


def _batch_boxes(c, seed):
    """the boxes of a batch, as coupled cases, with the seeds of their spheres
    (sizes belong to the case; positions to the seed)"""
    rng = np.random.default_rng(77 + c["boxes"])
    out = []
    for k in range(c["boxes"]):
        L = int(round(math.exp(rng.uniform(math.log(c["lo"]), math.log(c["hi"])))))
        eps = rng.uniform(c["eps_lo"], c["eps_hi"])
        out.append((_coupled(form=c["form"], nx=L, ny=L, nz=L, eps=eps, d=c["d"], h_c=1.0, n_int=4, n_dem=5,
                             steps=c["steps"]), 1000 * seed + k))
    return out


def _velocities():
    """the 19 lattice velocities, an order of this file's own"""
    return [(x, y, z) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1) if x * x + y * y + z * z <= 2]


def _weight(c):
    return {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}[c[0] ** 2 + c[1] ** 2 + c[2] ** 2]


def _fluid_inputs(c, seed):
    """A decaying flow: populations near equilibrium for a few velocity modes plus
    noise, a varying porosity and a force density; f [19][nz][ny][nx] in the order
    of _velocities()."""
    (nx, ny, nz), _ = _geometry(c)
    rng = np.random.default_rng(seed)
    z, y, x = torch.meshgrid(*(torch.arange(k, dtype=torch.float64, device=DEV) for k in (nz, ny, nx)), indexing="ij")
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))

    def modes(amp):
        v = torch.zeros_like(x)
        for _ in range(3):
            k = [2 * PI * rng.integers(1, 4) / m for m in (nx, ny, nz)]
            v += amp / 3 * torch.sin(k[0] * x + rng.uniform(0, 6.28)) * torch.sin(k[1] * y + rng.uniform(0, 6.28)) * \
                torch.cos(k[2] * z + rng.uniform(0, 6.28))
        return v

    u = [modes(0.03) for _ in range(3)]
    eps = 0.8 + modes(0.15)
    fpf = torch.stack([modes(1e-4) for _ in range(3)])
    f = []
    for q in _velocities():
        cu = q[0] * u[0] + q[1] * u[1] + q[2] * u[2]
        f.append(_weight(q) * (1 + 3 * cu + 4.5 * cu * cu / eps - 1.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2) / eps) *
                 (1 + 1e-4 * torch.randn(x.shape, dtype=torch.float64, device=DEV, generator=gen)))
    return torch.stack(f), eps, fpf


def prepare(case, seed):
    c = case
    if c["kind"] == "sort":
        rng = np.random.default_rng(seed)
        n, per = _geometry(c)
        x = np.minimum(rng.random((c["np"], 3)) * np.array(n, float), np.nextafter(np.array(n, float), 0))
        ids = rng.permutation(c["np"]).astype(np.int32)
        return dict(c=c, n=n, per=per, x=torch.from_numpy(x).to(DEV), ids=torch.from_numpy(ids).to(DEV))
    if c["kind"] == "batch":
        b = dps.Batch(c["form"])
        boxes = []
        for bc, s in _batch_boxes(c, seed):
            n, per = _geometry(bc)
            p = _coupled_inputs(bc, s)
            k = b.add_box(n, per, bc["tau"], len(p["x"]))
            b.add_particles(k, p["x"], p["d"], p["rho_p"], u=p["u"], w=p["w"])
            b.set_closure(k, **_closure(bc))
            boxes.append(k)
        return dict(c=c, batch=b, boxes=boxes)
    n, per = _geometry(c)
    if c["kind"] == "fluid":
        f, eps, fpf = _fluid_inputs(c, seed)
        order = {v: k for k, v in enumerate(_velocities())}
        planes = [order[tuple(int(t) for t in v)] for v in dps.lattice()[0]]
        dom = dps.Domain(n, per, c["tau"], c["form"])
        dom.write_pdfs(f[planes].cpu().numpy())
        dom.write_fields(eps_f=eps.cpu().numpy(), f_pf=fpf.cpu().numpy())
        return dict(c=c, dom=dom)
    p = _coupled_inputs(c, seed)
    dom = dps.Domain(n, per, c["tau"], c["form"], max_particles=len(p["x"]))
    dom.add_particles(p["x"], p["d"], p["rho_p"], u=p["u"], w=p["w"])
    dom.set_closure(**_closure(c))
    return dict(c=c, dom=dom)


# ---- one pass ------------------------------------------------------------------------
def _typed(c, out):
    """results in the form's own arithmetic type (the read-back calls return FP64)"""
    return out if c["form"] == "f64" else {k: v.astype(np.float32) for k, v in out.items()}


def run(state):
    c = state["c"]
    if c["kind"] == "sort":
        start, order = dps.op_cell_sort(state["n"], state["per"], state["x"], state["ids"])
        return dict(start=start, order=order)
    if c["kind"] == "batch":
        b = state["batch"]
        b.step(c["steps"])
        got = [b.read_particles(k) for k in state["boxes"]]
        return _typed(c, {k: np.concatenate([g[k] for g in got]) for k in ("x", "u", "w", "F")})
    dom = state["dom"]
    if c["kind"] == "fluid":
        dom.collide_stream(c["steps"])
        return _typed(c, dom.read_fields(("rho", "ubar")))
    dom.step(c["steps"])
    out = dom.read_particles()
    if c["nx"] * c["ny"] * c["nz"] <= 1 << 21:  # larger runs sample the particles every pass and the fluid rarely
        out["ubar"] = dom.read_fields(("ubar",))["ubar"]
    return _typed(c, out)


# ---- what one pass cannot do without ----------------------------------------------------
def _coupled_work(c, count):
    cells = c["nx"] * c["ny"] * c["nz"]
    s, sf = {"f64": (8, 8), "f32": (4, 4), "f16s": (2, 4)}[c["form"]]
    subs = c["n_int"] * c["n_dem"]
    rl = c["d"] + (c["h_c"])  # centres closer than this interact
    pairs = count * (count / cells) * 4.19 * rl ** 3 / 2
    # a step reads and writes the populations, eps_f and f_pf; a substep reads and
    # writes the particles' x, u, w and reads d, m and the frozen force
    per_step = cells * (38 * s + 8 * sf) + count * subs * 184
    flops = cells * (207 + 57 + 135) + count * c["n_int"] * 27 * 30 + subs * (32 * count + 75 * pairs)
    return c["steps"] * per_step, c["steps"] * flops


def work(case):
    c = case
    if c["kind"] == "sort":
        cells = c["nx"] * c["ny"] * c["nz"]
        return {"bytes": c["np"] * (24 + 4 + 4) + 4 * cells, "flops": 0}
    cells = 0 if c["kind"] == "batch" else c["nx"] * c["ny"] * c["nz"]
    if c["kind"] == "fluid":
        s, sf = {"f64": (8, 8), "f32": (4, 4), "f16s": (2, 4)}[c["form"]]
        return {"bytes": c["steps"] * cells * (38 * s + 4 * sf) + 32 * cells, "flops": c["steps"] * cells * 249}
    many = [b for b, _ in _batch_boxes(c, 0)] if c["kind"] == "batch" else [c]
    total = [0.0, 0.0]
    for b in many:
        count = max(1, b["eps"] * b["nx"] * b["ny"] * b["nz"] / (PI / 6 * b["d"] ** 3))
        by, fl = _coupled_work(b, count)
        total[0] += by + 96 * count
        total[1] += fl
    if c["kind"] == "coupled" and cells <= 1 << 21:
        total[0] += 24 * cells
    return {"bytes": total[0], "flops": total[1]}


# ---- the method in 64 bits ------------------------------------------------------------------
class _Lattice:
    """Cell fields are [nz][ny][nx] tensors; `at` reads a field at x + (cx, cy, cz)
    with periodic wrap, and at a wall either the cell itself (clamped) or, with
    `inside`, says where the neighbour lies in the box."""

    def __init__(self, n, per):
        self.n, self.per = n, per
        self.c = _velocities()
        self.w = [_weight(q) for q in self.c]
        self.index = []
        for a in range(3):
            i = torch.arange(n[a], device=DEV)
            self.index.append({o: (i + o) % n[a] if per[a] else (i + o).clamp(0, n[a] - 1) for o in (-1, 0, 1)})

    def at(self, f, c):
        for a in range(3):
            if c[a]:
                f = f.index_select(2 - a, self.index[a][c[a]])
        return f

    def inside(self, c):
        ok = torch.ones(self.n[::-1], dtype=torch.bool, device=DEV)
        for a in range(3):
            if c[a] and not self.per[a]:
                ok.select(2 - a, self.n[a] - 1 if c[a] > 0 else 0).fill_(False)
        return ok

    def gradient(self, f):
        g = [torch.zeros_like(f) for _ in range(3)]
        for c, w in zip(self.c, self.w):
            if any(c):
                v = self.at(f, c)
                for a in range(3):
                    if c[a]:
                        g[a] += 3 * w * c[a] * v
        return g

    def moments(self, f):
        rho, j = torch.zeros_like(f[0]), [torch.zeros_like(f[0]) for _ in range(3)]
        for q, c in enumerate(self.c):
            rho += f[q]
            for a in range(3):
                if c[a]:
                    j[a] += c[a] * f[q]
        return rho, j

    def equilibrium(self, rho, u, eps, q):
        c = self.c[q]
        cu = sum(c[a] * u[a] for a in range(3) if c[a]) if any(c) else torch.zeros_like(rho)
        uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        return cu, self.w[q] * rho * (1 + 3 * cu + 4.5 * cu * cu / eps - 1.5 * uu / eps)

    def collide_stream(self, f, eps, F, tau, eilers=0, smag=0):
        rho, j = self.moments(f)
        u = [(j[a] + 0.5 * F[a]) / rho for a in range(3)]
        te = torch.full_like(rho, tau)
        if eilers:
            r = ((1 - eps) / 0.64).clamp(0, 0.9)
            te = 0.5 + (tau - 0.5) * (1 + 1.25 * 0.64 * r / (1 - r)) ** 2
        if smag:
            Q = {}
            for q, c in enumerate(self.c):
                ne = f[q] - self.equilibrium(rho, u, eps, q)[1]
                for a in range(3):
                    for b in range(3):
                        if c[a] * c[b]:
                            Q[a, b] = Q.get((a, b), 0) + c[a] * c[b] * ne
            bar = torch.sqrt(2 * sum(v * v for v in Q.values()))
            te = te + 0.5 * (torch.sqrt(te * te + 0.18 * bar / rho) - te)
        uF = sum(u[a] * F[a] for a in range(3))
        post = []
        for q, c in enumerate(self.c):
            cu, feq = self.equilibrium(rho, u, eps, q)
            cF = sum(c[a] * F[a] for a in range(3) if c[a]) if any(c) else 0.0
            post.append(f[q] + (feq - f[q]) / te +
                        self.w[q] * (1 - 0.5 / te) * (3 * cF - 3 * uF / eps + 9 * cu * cF / eps))
        out = torch.empty_like(f)
        for q, c in enumerate(self.c):
            back = tuple(-v for v in c)
            v = self.at(post[q], back)
            ok = self.inside(back)
            out[q] = torch.where(ok, v, post[self.c.index(back)])
        return out


def _phi(r):
    r = r.abs()
    s = torch.where(r < 0.5, r, 1 - r)
    q = torch.sqrt((1 - 3 * s * s).clamp(min=0))
    return torch.where(r < 0.5, (1 + q) / 3, torch.where(r < 1.5, (5 - 3 * r - q) / 6, torch.zeros_like(r)))


class _Exact:
    """The coupled step (Algorithm 1) for one box."""

    def __init__(self, c, p):
        self.k, self.c = _closure(c), c
        self.n, self.per = _geometry(c)
        self.lat = _Lattice(self.n, self.per)
        t = lambda v: torch.from_numpy(np.array(v, np.float64)).to(DEV)  # noqa: E731
        self.x, self.u, self.w, self.d, self.rp = (t(p[s]) for s in ("x", "u", "w", "d", "rho_p"))
        self.V = PI / 6 * self.d ** 3
        self.m = self.rp * self.V
        self.tau = c["tau"]
        self.mu = (self.tau - 0.5) / 3
        shape = self.n[::-1]
        self.f = torch.stack([torch.full(shape, w, dtype=torch.float64, device=DEV) for w in self.lat.w])
        self.fpf = [torch.zeros(shape, dtype=torch.float64, device=DEV) for _ in range(3)]
        self.uprev = self.usub = None
        cells = self.n[0] * self.n[1] * self.n[2]
        g = self.k["g"]
        weight = float(((self.rp - 1) * self.V).sum())
        self.fb = [-weight * g[a] / (cells - float(self.V.sum())) if self.k["fb_mode"] == 1 else 0.0 for a in range(3)]
        self.L = torch.tensor(self.n, dtype=torch.float64, device=DEV)
        self.wrap = torch.tensor(self.per, dtype=torch.bool, device=DEV)
        self.F = torch.zeros_like(self.x)
        self.support()

    # the 27 cells and weights of every sphere, and eps_f
    def support(self):
        cell, wt = [], []
        for a in range(3):
            L = self.n[a]
            i = torch.floor(self.x[:, a]).long().clamp(0, L - 1)
            o = i[:, None] + torch.arange(-1, 2, device=DEV)
            v = _phi(o + 0.5 - self.x[:, a:a + 1])
            if not self.per[a]:
                v = torch.where((o >= 0) & (o < L), v, torch.zeros_like(v))
                v = v / v.sum(1, keepdim=True)
            cell.append(o % L if self.per[a] else o.clamp(0, L - 1))
            wt.append(v)
        nx, ny, _ = self.n
        self.idx = (cell[0][:, None, None, :] + nx * (cell[1][:, None, :, None] + ny * cell[2][:, :, None, None])).reshape(-1, 27)
        self.D = (wt[0][:, None, None, :] * wt[1][:, None, :, None] * wt[2][:, :, None, None]).reshape(-1, 27)
        self.eps = (1 - self.spread(self.V)).clamp(min=self.k["eps_min"])

    def spread(self, v):
        out = torch.zeros(self.n[0] * self.n[1] * self.n[2], dtype=torch.float64, device=DEV)
        for k in range(27):
            out.index_add_(0, self.idx[:, k], self.D[:, k] * v)
        return out.reshape(self.n[::-1])

    def interp(self, f):
        f = f.reshape(-1)
        return sum(self.D[:, k] * f[self.idx[:, k]] for k in range(27))

    def image(self, dx):
        return torch.where(self.wrap, dx - self.L * torch.round(dx / self.L), dx)

    # candidate pairs i < j within the interaction range plus a margin
    def pairs(self):
        reach = float(self.d.max()) + self.k["h_c"] + 0.35
        nb = [int(self.n[a] / reach) for a in range(3)]
        N = len(self.x)
        if N < 3000 or any(nb[a] < 3 for a in range(3)):
            i, j = torch.triu_indices(N, N, 1, device=DEV)
            keep = (self.image(self.x[j] - self.x[i]).norm(dim=1) < reach)
            return i[keep], j[keep]
        b = [(self.x[:, a] * (nb[a] / self.n[a])).long().clamp(0, nb[a] - 1) for a in range(3)]
        key = b[0] + nb[0] * (b[1] + nb[1] * b[2])
        order = torch.argsort(key)
        start = torch.zeros(nb[0] * nb[1] * nb[2] + 1, dtype=torch.long, device=DEV)
        start[1:] = torch.cumsum(torch.bincount(key, minlength=len(start) - 1), 0)
        ii, jj = [], []
        for o in [(x, y, z) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)]:
            if o < (0, 0, 0):
                continue
            t = [b[a] + o[a] for a in range(3)]
            ok = torch.ones(N, dtype=torch.bool, device=DEV)
            for a in range(3):
                if self.per[a]:
                    t[a] = t[a] % nb[a]
                else:
                    ok &= (t[a] >= 0) & (t[a] < nb[a])
                    t[a] = t[a].clamp(0, nb[a] - 1)
            k = t[0] + nb[0] * (t[1] + nb[1] * t[2])
            cnt = torch.where(ok, start[k + 1] - start[k], torch.zeros_like(k))
            i = torch.repeat_interleave(torch.arange(N, device=DEV), cnt)
            at = torch.arange(len(i), device=DEV) - torch.repeat_interleave(torch.cumsum(cnt, 0) - cnt, cnt)
            j = order[start[k][i] + at]
            keep = (i < j) if o == (0, 0, 0) else torch.ones_like(i, dtype=torch.bool)
            i, j = i[keep], j[keep]
            keep = self.image(self.x[j] - self.x[i]).norm(dim=1) < reach
            ii.append(i[keep])
            jj.append(j[keep])
        return torch.cat(ii), torch.cat(jj)

    # force on the first partner and n x F_t, given unit normals and distances
    def interact(self, n, dist, sumr, ui, uj, spin, mij, dm, dt):
        k = self.k
        le = math.log(k["e_n"])
        kn, xi = mij * (PI ** 2 + le ** 2) / k["T_c"] ** 2, -2 * le * mij / k["T_c"]
        F, Tq = torch.zeros_like(n), torch.zeros_like(n)
        over = torch.nonzero(sumr - dist > 0)[:, 0]
        if len(over):
            nn = n[over]
            ur = ui[over] - uj[over] + torch.linalg.cross(spin[over], nn)
            un = (ur * nn).sum(1, keepdim=True)
            ut = ur - un * nn
            Fn = -(kn * (sumr - dist))[over, None] * nn - xi[over, None] * un * nn
            ua = ut.norm(dim=1, keepdim=True)
            mag = torch.minimum(k["mu_c"] * Fn.norm(dim=1, keepdim=True), xi[over, None] * ua)
            Ft = torch.where(ua > 0, -mag * ut / ua.clamp(min=1e-300), torch.zeros_like(ut))
            F[over] = Fn + Ft
            Tq[over] = torch.linalg.cross(nn, Ft)
        h = dist - sumr
        near = torch.nonzero((h >= 0) & (h < k["h_c"]))[:, 0]
        if len(near):
            hh, dmn, nn = h[near].clamp(min=k["h_min"]), dm[near], n[near]
            Lg = torch.log(dmn / (2 * hh))
            sq = 1.5 * PI * self.mu * dmn * (dmn / (4 * hh) + 18 / 40 * Lg + 9 / 84 * hh / dmn * Lg)
            sh = 0.5 * PI * self.mu * dmn * Lg
            cap = k["lub_cap"] * mij[near] / dt
            sq, sh = (torch.minimum(v.clamp(min=0), cap)[:, None] for v in (sq, sh))
            ur = ui[near] - uj[near]
            un = (ur * nn).sum(1, keepdim=True)
            F[near] += -sq * un * nn - sh * (ur - un * nn)
        return F, Tq

    def dem(self, dt):
        k = self.k
        i, j = self.pairs()
        for _ in range(k["n_dem"]):
            F, T = self.F.clone(), torch.zeros_like(self.F)
            dx = self.image(self.x[j] - self.x[i])
            dist = dx.norm(dim=1)
            sumr = 0.5 * (self.d[i] + self.d[j])
            on = torch.nonzero((dist < sumr + k["h_c"]) & (dist > 0))[:, 0]
            a, b, dist, sumr = i[on], j[on], dist[on], sumr[on]
            n = dx[on] / dist[:, None]
            mij = self.m[a] * self.m[b] / (self.m[a] + self.m[b])
            dm = 2 * self.d[a] * self.d[b] / (self.d[a] + self.d[b])
            spin = 0.5 * (self.d[a, None] * self.w[a] + self.d[b, None] * self.w[b])
            Fp, Tp = self.interact(n, dist, sumr, self.u[a], self.u[b], spin, mij, dm, dt)
            F.index_add_(0, a, Fp)
            F.index_add_(0, b, -Fp)
            T.index_add_(0, a, 0.5 * self.d[a, None] * Tp)
            T.index_add_(0, b, 0.5 * self.d[b, None] * Tp)
            for ax in range(3):
                if self.per[ax]:
                    continue
                for side in (0, 1):
                    dist = self.x[:, ax] if side == 0 else self.n[ax] - self.x[:, ax]
                    n = torch.zeros_like(self.x)
                    n[:, ax] = 2 * side - 1
                    Fw, Tw = self.interact(n, dist, 0.5 * self.d, self.u, torch.zeros_like(self.u),
                                           0.5 * self.d[:, None] * self.w, self.m, 2 * self.d, dt)
                    F += Fw
                    T += 0.5 * self.d[:, None] * Tw
            self.u = self.u + dt * F / self.m[:, None]
            self.w = self.w + dt * T / (self.m * self.d ** 2 / 10)[:, None]
            x = self.x + dt * self.u
            self.x = torch.where(self.wrap, x - self.L * torch.floor(x / self.L), x)

    def uf(self, rho, j, F):
        return [(j[a] + 0.5 * F[a]) / rho / self.eps for a in range(3)]

    def step(self):
        k, lat = self.k, self.lat
        g, dts = k["g"], 1.0 / k["n_int"]
        rho, j = lat.moments(self.f)
        uD = self.uf(rho, j, [self.eps * self.fb[a] + self.fpf[a] for a in range(3)])
        prev = self.uprev or uD
        DuDt = [uD[b] - prev[b] + sum(uD[a] * gr for a, gr in enumerate(lat.gradient(uD[b]))) for b in range(3)]
        self.uprev = uD
        gradP = [v / 3 for v in lat.gradient(rho)]
        total = [torch.zeros_like(rho) for _ in range(3)]
        for _ in range(k["n_int"]):
            dudt = (self.u - self.usub) / dts if self.usub is not None else torch.zeros_like(self.u)
            self.usub = self.u
            Fa = 0.5 * self.V[:, None] * (torch.stack([self.interp(v) for v in DuDt], 1) - dudt)
            if k["lift"]:
                uf = self.uf(rho, j, [self.eps * self.fb[a] for a in range(3)])
                gr = [lat.gradient(v) for v in uf]  # gr[b][a] = d_a u_b
                curl = [gr[2][1] - gr[1][2], gr[0][2] - gr[2][0], gr[1][0] - gr[0][1]]
                om = torch.stack([self.interp(v) for v in curl], 1)
                du = torch.stack([self.interp(v) for v in uf], 1) - self.u
                wn = om.norm(dim=1, keepdim=True)
                lift = 1.61 * (self.d ** 2)[:, None] * torch.sqrt(self.mu / wn.clamp(min=1e-300)) * torch.linalg.cross(du, om)
                Fa = Fa + torch.where(wn > 0, lift, torch.zeros_like(lift))
            fpf = [-self.spread(Fa[:, a]) for a in range(3)]
            uf = self.uf(rho, j, [self.eps * self.fb[a] + fpf[a] for a in range(3)])
            du = torch.stack([self.interp(v) for v in uf], 1) - self.u
            gP = torch.stack([self.interp(v) for v in gradP], 1)
            ef = self.interp(self.eps)
            ep = 1 - ef
            Re = ef * self.d * du.norm(dim=1) / self.mu
            e1 = 1 - ep
            cd = e1 * ((1 + 0.15 * Re ** 0.687) / e1 ** 3 + 5.81 * ep / e1 ** 3 +
                       0.48 * ep.clamp(min=0) ** (1 / 3) / e1 ** 4 + ep ** 3 * Re * (0.95 + 0.61 * ep ** 3 / e1 ** 2))
            Fd = (3 * PI * self.d * self.mu * e1 * cd)[:, None] * du
            grav = ((self.rp - 1) * self.V)[:, None] * torch.tensor(g, dtype=torch.float64, device=DEV)
            self.F = Fd - self.V[:, None] * gP + Fa + grav
            for a in range(3):
                total[a] += fpf[a] - self.spread(Fd[:, a])
            self.dem(dts / k["n_dem"])
            self.support()
        self.fpf = [v * dts for v in total]
        F = [self.fpf[a] + self.eps * self.fb[a] for a in range(3)]
        self.f = lat.collide_stream(self.f, self.eps, F, self.tau, k["eilers"], k["smagorinsky"])

    def ubar(self):
        rho, j = self.lat.moments(self.f)
        return torch.stack([((j[a] + 0.5 * (self.fpf[a] + self.eps * self.fb[a])) / rho).reshape(-1) for a in range(3)])


def exact(case, seed):
    c = case
    if c["kind"] == "sort":
        return None  # whole numbers, compared bit for bit
    if c["kind"] == "fluid":
        n, per = _geometry(c)
        f, eps, fpf = _fluid_inputs(c, seed)
        lat = _Lattice(n, per)
        for _ in range(c["steps"]):
            f = lat.collide_stream(f, eps, fpf, c["tau"])
        rho, j = lat.moments(f)
        ub = torch.stack([((j[a] + 0.5 * fpf[a]) / rho).reshape(-1) for a in range(3)])
        return dict(rho=rho.reshape(-1), ubar=ub)
    many = _batch_boxes(c, seed) if c["kind"] == "batch" else [(c, seed)]
    got = []
    for bc, s in many:
        e = _Exact(bc, _coupled_inputs(bc, s))
        for _ in range(c["steps"]):
            e.step()
        got.append(e)
    out = dict(x=torch.cat([e.x for e in got]), u=torch.cat([e.u for e in got]), w=torch.cat([e.w for e in got]),
               F=torch.cat([e.F for e in got]))
    if c["kind"] == "coupled" and c["nx"] * c["ny"] * c["nz"] <= 1 << 21:
        out["ubar"] = got[0].ubar()
    return out
