"""The work a user of this library has it do, as cases that can be timed and checked one by one.

Every case goes through the public binding (``paper_1907_00890_gb300.vofp``).  ``prepare`` makes what a flow code has
in hand before the call -- fields on the GPU (host memory for the host-buffer step), a plan, a batch or a server --
``run`` makes one call as that code would, ``exact`` evaluates the same result with plain torch in FP64 (dense
eigenvector products in x and y, Thomas elimination in z), ``work`` counts what the call cannot do without.

Projections work in place on the velocity; a flow code's predictor writes u* anew before each of them, and the
copy of u* into the projected buffer at the start of those passes stands for that.
"""
import math

import numpy as np
import torch

from paper_1907_00890_gb300 import synth, vofp

F64 = torch.float64
PREC = {"fp64": vofp.FP64, "mixed": vofp.MIXED, "ff": vofp.FF}
RHO1, RHO2 = 100.0, 1.0  # density ratio 100
BCS = ("P", "NN", "DD", "ND", "DN")


def _case(name, kind, n, bc, prec="fp64", **more):
    c = {"name": name, "kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "bcx": bc[0], "bcy": bc[1], "bcz": bc[2],
         "prec": prec, "stretched": False, "youngs": False}
    c.update(more)
    return c


def listed():
    ppn = ("P", "P", "NN")
    return [
        # the smallest call: one projection of a 32^3 run, where launches and latency count
        _case("project_32", "project", (32, 32, 32), ppn),
        # the ordinary time step: projection and liquid-velocity extension of a droplet, plain FP64
        _case("step_128", "step", (128, 128, 128), ppn),
        # the same step in the direct FP32-pair precision
        _case("step_128_ff", "step", (128, 128, 128), ppn, "ff"),
        # the same step called by a code that keeps its fields in (pinned) host memory
        _case("step_128_host", "step_host", (128, 128, 128), ppn),
        # the largest single solve: stretched z, FP32 transforms with FP64 refinement
        _case("project_512_mixed", "project", (512, 512, 512), ppn, "mixed", stretched=True),
        # the settling-droplet grid, periodic on every axis
        _case("step_320x320x640", "step", (320, 320, 640), ("P", "P", "P")),
        # one pressure or potential solve in a walled container, sides of no power of two
        _case("poisson_250x150x128_walls", "poisson", (250, 150, 128), ("NN", "NN", "ND"), stretched=True),
        # the variable-density pressure step
        _case("vd_128", "vd", (128, 128, 128), ppn),
        # an extension alone, Youngs' gradient, small ragged grid with walls
        _case("extend_96x80x72_youngs", "extend", (96, 80, 72), ("NN", "NN", "DN"), youngs=True),
        # the volume-fraction update with the interface velocity
        _case("vof_128", "vof", (128, 128, 128), ppn),
        # an ensemble of independent runs with uneven grids, one batched call
        _case("batch_64_mixed", "batch", (0, 0, 0), ppn, "mixed", count=64, sizes=synth.BASE_SEED + 4),
        # a burst of served projection requests with uneven grids, plans resident after the first
        _case("serve_24_ff", "serve", (0, 0, 0), ppn, "ff", count=24, sizes=synth.BASE_SEED + 5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["project", "project", "poisson", "poisson", "step", "step", "step_host", "vd", "extend", "vof",
                       "batch", "serve"])
    prec = rng.choice(["fp64", "fp64", "mixed", "ff"])
    if kind in ("batch", "serve"):
        c = _case("", kind, (0, 0, 0), ("P", "P", "NN"), rng.choice(["mixed", "ff"]), count=rng.randint(4, 24),
                  sizes=rng.randrange(1 << 20))
    else:
        while True:
            # any length, or one of the sides with small factors that flow codes prefer
            n = [_log_int(rng, 16, 384) if rng.random() < 0.5 else
                 rng.choice([32, 48, 64, 96, 128, 160, 192, 256, 320, 384]) for _ in range(3)]
            if n[0] * n[1] * n[2] <= 12 << 20:
                break
        bc = [rng.choice(("P", "P", "P", "NN", "NN", "DD", "ND", "DN")) for _ in range(2)] + [rng.choice(BCS)]
        c = _case("", kind, n, bc, prec, stretched=bc[2] != "P" and rng.random() < 0.3, youngs=rng.random() < 0.2)
    del c["name"]
    return c


# ---- what a user has in hand ------------------------------------------------------------------------------------

def _sizes(case):
    if case["kind"] == "batch":
        return synth.batch_sizes(case["count"], seed=case["sizes"])
    if case["kind"] == "serve":
        return synth.serve_sizes(case["count"], seed=case["sizes"])
    return [(case["nx"], case["ny"], case["nz"])]


def _bc(case):
    return (case["bcx"], case["bcy"], case["bcz"])


def _dz(case, n):
    return synth.stretched_dz(n[2]) if case["stretched"] else synth.uniform_dz(n[2])


def _plan(case, n):
    return vofp.Plan(n, 1.0 / n[0], 1.0 / n[1], _dz(case, n), _bc(case), prec=PREC[case["prec"]],
                     max_refine=0 if case["prec"] == "ff" else 3, grad_mode=1 if case["youngs"] else 0)


def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + salt)
    return g


def _views(flat, shapes):
    out, o = [], 0
    for s in shapes:
        m = s[0] * s[1] * s[2]
        out.append(flat[o:o + m].view(s))
        o += m
    return out


def _close_walls(views, bc):
    for axis in range(3):
        if bc[axis] != "P":
            views[axis].select(2 - axis, 0).zero_()
            views[axis].select(2 - axis, -1).zero_()


def _noise(n, bc, seed, salt, sigma):
    """N(0, sigma) face velocities (u, v, w in one buffer), zero on walls."""
    shapes = vofp.face_shapes(n, bc)
    flat = torch.empty(sum(a * b * c for a, b, c in shapes), dtype=F64, device="cuda")
    flat.normal_(0.0, sigma, generator=_gen(seed, salt))
    views = _views(flat, shapes)
    _close_walls(views, bc)
    return flat, views


def _droplet(case, n, seed):
    """Liquid indicator of a sphere (radius 0.15, tanh profile 1.5 cells wide) and the evaporation rate around 1."""
    bc, dz = _bc(case), _dz(case, n)
    c = 0.5 + 0.2 * (torch.rand(3, dtype=F64, device="cuda", generator=_gen(seed, 7)) - 0.5)
    zf = np.concatenate([[0.0], np.cumsum(dz)])
    pos = [torch.as_tensor((np.arange(n[a]) + 0.5) / n[a] if a < 2 else 0.5 * (zf[:-1] + zf[1:]), device="cuda")
           for a in range(3)]
    d = [pos[a] - c[a] for a in range(3)]
    d = [x - torch.round(x) if bc[a] == "P" else x for a, x in enumerate(d)]
    r = torch.sqrt(d[2][:, None, None] ** 2 + d[1][None, :, None] ** 2 + d[0][None, None, :] ** 2)
    C = 0.5 * (1.0 - torch.tanh((r - 0.15) / (1.5 / n[0])))
    mdot = 1.0 + 0.05 * torch.randn(C.shape, dtype=F64, device="cuda", generator=_gen(seed, 8))
    return C, mdot, c


def _swirl(case, n, seed, centre):
    """Solid-body swirl about the droplet's axis plus N(0, 0.1) noise, zero on walls."""
    bc = _bc(case)
    flat, (u, v, w) = _noise(n, bc, seed, 9, 0.1)
    yc = (torch.arange(n[1], dtype=F64, device="cuda") + 0.5) / n[1]
    xc = (torch.arange(n[0], dtype=F64, device="cuda") + 0.5) / n[0]
    u -= 2.0 * (yc - centre[1])[None, :, None]
    v += 2.0 * (xc - centre[0])[None, None, :]
    _close_walls((u, v, w), bc)
    return flat


class _Batch:
    def __init__(self, plans):
        self.plans = plans
        self.handle = vofp.vofp_batch_create([p.handle for p in plans])

    def __del__(self):
        vofp.vofp_batch_destroy(self.handle)


class _Server:
    def __init__(self, prec, inflight):
        o = vofp.vofp_opts_default()
        o.prec, o.max_refine = prec, 0 if prec == vofp.FF else 3
        self.handle = vofp.vofp_server_create(6 << 30, inflight, o)

    def __del__(self):
        vofp.vofp_server_destroy(self.handle)


def prepare(case, seed):
    kind, bc = case["kind"], _bc(case)
    s = {"case": case}
    if kind in ("batch", "serve"):
        sizes = _sizes(case)
        star, p, parts = [], [], []
        for i, n in enumerate(sizes):
            star.append(_noise(n, bc, seed, 100 + i, 1.0)[0])
            p.append(torch.empty(n[0] * n[1] * n[2], dtype=F64, device="cuda"))
        s["star"], s["p"] = torch.cat(star), torch.cat(p)
        s["vel"] = torch.empty_like(s["star"])
        ov = op = 0
        for n, a, b in zip(sizes, star, p):
            parts.append((n, _views(s["vel"][ov:ov + a.numel()], vofp.face_shapes(n, bc)),
                          s["p"][op:op + b.numel()].view(n[2], n[1], n[0])))
            ov += a.numel()
            op += b.numel()
        s["parts"] = parts
        if kind == "batch":
            s["batch"] = _Batch([_plan(case, n) for n in sizes])
        else:
            s["server"] = _Server(PREC[case["prec"]], 32)
        return s
    n = _sizes(case)[0]
    cells = (n[2], n[1], n[0])
    s["plan"] = _plan(case, n)
    if kind == "poisson":
        s["f"] = torch.randn(cells, dtype=F64, device="cuda", generator=_gen(seed, 1))
        s["p"] = torch.empty_like(s["f"])
        return s
    if kind == "project":
        s["star"] = _noise(n, bc, seed, 2, 1.0)[0]
        s["vel"] = torch.empty_like(s["star"])
        s["uvw"] = _views(s["vel"], vofp.face_shapes(n, bc))
        s["p"] = torch.empty(cells, dtype=F64, device="cuda")
        return s
    C, mdot, centre = _droplet(case, n, seed)
    s["C"], s["mdot"] = C, mdot
    if kind == "vof":
        # the interface velocity's size and a step at a Courant number of one half
        flat, s["ug"] = _noise(n, bc, seed, 3, 0.5)
        s["dt"] = float(0.5 / (flat.abs().max() * (n[0] + n[1] + float(1.0 / _dz(case, n).min()))))
        s["out"] = torch.empty_like(C)
        s["work"] = torch.empty((2,) + cells, dtype=F64, device="cuda")
        return s
    s["star"] = _swirl(case, n, seed, centre)
    shapes = vofp.face_shapes(n, bc)
    if kind == "step_host":
        s["in"] = [t.cpu().pin_memory() for t in _views(s.pop("star"), shapes)]
        s["C"], s["mdot"] = C.cpu().pin_memory(), mdot.cpu().pin_memory()
        s["out"] = [torch.empty(sh, dtype=F64, pin_memory=True) for sh in shapes + (cells,) + shapes]
        return s
    s["vel"] = torch.empty_like(s["star"])
    s["uvw"] = _views(s["vel"], shapes)
    s["p"] = torch.empty(cells, dtype=F64, device="cuda")
    if kind == "vd":
        g = _gen(seed, 4)
        s["pn"] = 0.1 * C + 0.01 * torch.randn(cells, dtype=F64, device="cuda", generator=g)
        s["pm"] = 0.95 * s["pn"]
    else:
        s["ue"] = _views(torch.empty_like(s["star"]), shapes)
        s["ug"] = _views(torch.empty_like(s["star"]), shapes)
        if kind == "extend":
            s["star"] = _views(s["star"], shapes)
    return s


def run(s):
    kind = s["case"]["kind"]
    if kind == "poisson":
        vofp.vofp_poisson_solve(s["plan"].handle, s["f"], s["p"])
        return {"p": s["p"]}
    if kind == "vof":
        vofp.vofp_vof_update(s["plan"].handle, s["C"], *s["ug"], s["dt"], s["out"], s["work"])
        return {"C": s["out"]}
    if kind == "extend":
        vofp.vofp_extend_liquid_velocity(s["plan"].handle, *s["star"], s["C"], s["mdot"], RHO1, RHO2, *s["ue"], *s["ug"],
                                         phi=s["p"])
        return {"ue": s["ue"], "ug": s["ug"], "phi": s["p"]}
    if kind == "step_host":
        o = s["out"]
        vofp.vofp_project_extend_host(s["plan"].handle, *s["in"], s["C"], s["mdot"], RHO1, RHO2, 1.0, *o)
        return {"u": o[:3], "p": o[3], "ug": o[4:]}
    s["vel"].copy_(s["star"])
    if kind == "project":
        vofp.vofp_project(s["plan"].handle, *s["uvw"], None, 1.0, s["p"])
        return {"u": s["uvw"], "p": s["p"]}
    if kind == "step":
        vofp.vofp_project_extend(s["plan"].handle, *s["uvw"], s["C"], s["mdot"], RHO1, RHO2, 1.0, s["p"], *s["ue"],
                                 *s["ug"])
        return {"u": s["uvw"], "p": s["p"], "ue": s["ue"], "ug": s["ug"]}
    if kind == "vd":
        vofp.vofp_project_vd(s["plan"].handle, *s["uvw"], None, s["C"], s["pn"], s["pm"], 1e-3, 1e-3, RHO1, RHO2, s["p"])
        return {"u": s["uvw"], "p": s["p"]}
    if kind == "batch":
        vel = list(zip(*[v for _, v, _ in s["parts"]]))
        vofp.vofp_batch_project(s["batch"].handle, *vel, None, [1.0] * len(s["parts"]), [p for _, _, p in s["parts"]])
        return {"u": s["vel"], "p": s["p"]}
    # served requests run on the server's own streams: the caller waits for its fields, submits, and waits
    torch.cuda.current_stream().synchronize()
    h = s["server"].handle
    tickets = [vofp.vofp_server_submit(h, n, 1.0 / n[0], 1.0 / n[1], _dz(s["case"], n), _bc(s["case"]), *v, p=p)
               for n, v, p in s["parts"]]
    for t in tickets:
        vofp.vofp_server_wait(h, t)
    return {"u": s["vel"], "p": s["p"]}


def work(case):
    kind, bc = case["kind"], _bc(case)
    by = fl = 0.0
    for n in _sizes(case):
        cells = float(n[0]) * n[1] * n[2]
        faces = float(sum(a * b * c for a, b, c in vofp.face_shapes(n, bc)))
        # real transforms of x and y there and back (2.5 m log2 m a line), three operations a row of z each way
        solve = cells * (5.0 * math.log2(max(2, n[0])) + 5.0 * math.log2(max(2, n[1])) + 6.0)
        b, f = {
            "poisson": (2 * cells, solve),
            "project": (2 * faces + cells, solve + 7 * cells + 2 * faces),
            "batch": (2 * faces + cells, solve + 7 * cells + 2 * faces),
            "serve": (2 * faces + cells, solve + 7 * cells + 2 * faces),
            "vd": (2 * faces + 4 * cells, solve + 7 * cells + 12 * faces),
            "extend": (3 * faces + 3 * cells, solve + 15 * cells + 6 * faces),
            "step": (4 * faces + 3 * cells, 2 * solve + 22 * cells + 8 * faces),
            "step_host": (3 * faces + 3 * cells, 2 * solve + 22 * cells + 8 * faces),
            "vof": (faces + 2 * cells, 30 * cells),
        }[kind]
        by += 8 * b
        fl += f
    return {"bytes": by, "flops": fl}


# ---- the same results in plain torch, FP64 ----------------------------------------------------------------------

def _modes(n, bc):
    """Orthonormal eigenvectors (columns) of the 1-D second difference and its eigenvalues times h^2."""
    j, m = np.arange(n)[:, None], np.arange(n)[None, :]
    if bc == "P":
        k = (m + 1) // 2
        a = 2.0 * np.pi * ((j * k) % n) / n
        q = np.where((m % 2 == 1) | (m == 0), np.cos(a), np.sin(a))
        lam = -4.0 * np.sin(np.pi * k[0] / n) ** 2
    else:
        k = {"NN": 2 * m, "DD": 2 * m + 2, "ND": 2 * m + 1, "DN": 2 * m + 1}[bc]  # argument pi k (2j+1) / (4n)
        a = np.pi * ((k * (2 * j + 1)) % (8 * n)) / (4.0 * n)
        q = np.cos(a) if bc in ("NN", "ND") else np.sin(a)
        lam = -4.0 * np.sin(np.pi * k[0] / (4.0 * n)) ** 2
    q = q / np.sqrt((q * q).sum(0))
    return torch.as_tensor(q, device="cuda"), torch.as_tensor(lam, device="cuda")


class _Exact:
    def __init__(self, case, n):
        self.n, self.bc = n, _bc(case)
        self.h = [torch.full((n[0],), 1.0 / n[0], dtype=F64, device="cuda"),
                  torch.full((n[1],), 1.0 / n[1], dtype=F64, device="cuda"),
                  torch.as_tensor(_dz(case, n), device="cuda")]
        self.youngs = case["youngs"]
        self.vol = self.h[2][:, None, None]
        self.singular = all(b in ("P", "NN") for b in self.bc)

    def shaped(self, a, axis):
        return a.view([-1 if d == 2 - axis else 1 for d in range(3)])

    def low_high(self, q, axis):
        """Values of a cell field on both sides of each face; beyond a bounded end the end cell."""
        d = 2 - axis
        if self.bc[axis] == "P":
            return torch.roll(q, 1, d), q
        m = self.n[axis]
        return (torch.cat([q.narrow(d, 0, 1), q], d), torch.cat([q, q.narrow(d, m - 1, 1)], d))

    def grad(self, p, axis):
        d, m, h = 2 - axis, self.n[axis], self.h[axis]
        if self.bc[axis] == "P":
            return (p - torch.roll(p, 1, d)) / self.shaped(0.5 * (h + torch.roll(h, 1)), axis)
        out = torch.zeros(tuple(m + 1 if e == d else p.shape[e] for e in range(3)), dtype=F64, device="cuda")
        if m > 1:
            out.narrow(d, 1, m - 1).copy_((p.narrow(d, 1, m - 1) - p.narrow(d, 0, m - 1)) /
                                          self.shaped(0.5 * (h[1:] + h[:-1]), axis))
        if self.bc[axis] in ("DD", "DN"):
            out.narrow(d, 0, 1).copy_(2.0 * p.narrow(d, 0, 1) / h[0])
        if self.bc[axis] in ("DD", "ND"):
            out.narrow(d, m, 1).copy_(-2.0 * p.narrow(d, m - 1, 1) / h[-1])
        return out

    def diff(self, f, axis):
        d, m = 2 - axis, self.n[axis]
        hi = torch.roll(f, -1, d) if self.bc[axis] == "P" else f.narrow(d, 1, m)
        lo = f if self.bc[axis] == "P" else f.narrow(d, 0, m)
        return (hi - lo) / self.shaped(self.h[axis], axis)

    def div(self, f):
        return self.diff(f[0], 0) + self.diff(f[1], 1) + self.diff(f[2], 2)

    def mean(self, q):
        return (q * self.vol).sum() / (self.vol.sum() * self.n[0] * self.n[1])

    def direct(self, f):
        n, bc = self.n, self.bc
        qx, lx = _modes(n[0], bc[0])
        qy, ly = _modes(n[1], bc[1])
        lam = (ly * n[1] ** 2)[:, None] + (lx * n[0] ** 2)[None, :]
        g = torch.matmul(qy.T, torch.matmul(f, qx))
        if bc[2] == "P":  # (uniform widths on a periodic axis)
            qz, lz = _modes(n[2], "P")
            g = torch.tensordot(qz.T, g, dims=1)
            den = lam[None] + (lz * n[2] ** 2)[:, None, None]
            if self.singular:
                den[0, 0, 0] = 1.0
                g[0, 0, 0] = 0.0
            g = torch.tensordot(qz, g / den, dims=1)
        else:
            w = self.h[2].cpu().numpy()
            hc = np.concatenate([[w[0]], 0.5 * (w[1:] + w[:-1]), [w[-1]]])
            lo, hi = 1.0 / (w * hc[:-1]), 1.0 / (w * hc[1:])
            b = -(lo + hi)
            b[0] += lo[0] if bc[2] in ("NN", "ND") else -lo[0]
            b[-1] += hi[-1] if bc[2] in ("NN", "DN") else -hi[-1]
            cp = torch.empty_like(g)
            for k in range(n[2]):
                den = lam + b[k]
                if k:
                    den = den - lo[k] * cp[k - 1]
                    g[k] -= lo[k] * g[k - 1]
                if self.singular and k == 0:
                    den[0, 0] = 1.0
                cp[k] = (hi[k] if k < n[2] - 1 else 0.0) / den
                g[k] /= den
                if self.singular and k == 0:  # pinned: p_0 = 0 in the mean mode
                    cp[k, 0, 0] = 0.0
                    g[k, 0, 0] = 0.0
            for k in range(n[2] - 2, -1, -1):
                g[k] -= cp[k] * g[k + 1]
        return torch.matmul(torch.matmul(qy, g), qx.T)

    def solve(self, f):
        if self.singular:
            f = f - self.mean(f)
        p = self.direct(f)
        for _ in range(2):
            r = f - self.div([self.grad(p, a) for a in range(3)])
            p = p + self.direct(r - self.mean(r) if self.singular else r)
        return p - self.mean(p) if self.singular else p

    def project(self, vel, src, dt):
        p = self.solve((self.div(vel) - (0.0 if src is None else src)) / dt)
        return [vel[a] - dt * self.grad(p, a) for a in range(3)], p

    def shift(self, q, axis, by):
        d, m = 2 - axis, self.n[axis]
        if self.bc[axis] == "P":
            return torch.roll(q, -by, d)
        i = torch.clamp(torch.arange(m, device="cuda") + by, 0, m - 1)
        return q.index_select(d, i)

    def grad_c(self, C):
        out = []
        for a in range(3):
            h = self.h[a]
            if self.bc[a] == "P":
                dist = 0.5 * (h + torch.roll(h, 1))
                dist = torch.cat([dist, dist[:1]])
            else:
                dist = torch.cat([h[:1], 0.5 * (h[1:] + h[:-1]), h[-1:]])
            if not self.youngs:
                out.append((self.shift(C, a, 1) - self.shift(C, a, -1)) / self.shaped(dist[1:] + dist[:-1], a))
                continue
            q = C
            for t in range(3):
                if t != a:
                    q = 0.25 * self.shift(q, t, -1) + 0.5 * q + 0.25 * self.shift(q, t, 1)
            out.append(0.5 * ((q - self.shift(q, a, -1)) / self.shaped(dist[:-1], a) +
                              (self.shift(q, a, 1) - q) / self.shaped(dist[1:], a)))
        return out

    def geometry(self, C, mdot):
        g = self.grad_c(C)
        m = torch.sqrt(g[0] ** 2 + g[1] ** 2 + g[2] ** 2)
        on = (torch.minimum(C, 1.0 - C) >= 1e-8) & (m > 0)
        one = torch.where(m > 0, m, torch.ones_like(m))
        return mdot * (1.0 / RHO2 - 1.0 / RHO1) * m, [torch.where(on, -x / one, torch.zeros_like(x)) for x in g]

    def face(self, q, axis):
        lo, hi = self.low_high(q, axis)
        return 0.5 * (lo + hi)

    def extend(self, vel, s, nrm, mdot):
        phi = self.solve(s)
        ue = [vel[a] - self.grad(phi, a) for a in range(3)]
        return ue, [ue[a] - self.face(mdot, a) / RHO1 * self.face(nrm[a], a) for a in range(3)], phi


def exact(case, seed):
    kind, bc = case["kind"], _bc(case)
    if kind in ("batch", "serve"):
        us, ps = [], []
        for i, n in enumerate(_sizes(case)):
            vel, p = _Exact(case, n).project(_noise(n, bc, seed, 100 + i, 1.0)[1], None, 1.0)
            us += [v.reshape(-1) for v in vel]
            ps.append(p.reshape(-1))
        return {"u": torch.cat(us), "p": torch.cat(ps)}
    n = _sizes(case)[0]
    e = _Exact(case, n)
    if kind == "poisson":
        return {"p": e.solve(torch.randn((n[2], n[1], n[0]), dtype=F64, device="cuda", generator=_gen(seed, 1)))}
    if kind == "project":
        vel, p = e.project(_noise(n, bc, seed, 2, 1.0)[1], None, 1.0)
        return {"u": vel, "p": p}
    C, mdot, centre = _droplet(case, n, seed)
    if kind == "vof":
        flat, ug = _noise(n, bc, seed, 3, 0.5)
        dt = float(0.5 / (flat.abs().max() * (n[0] + n[1] + float(1.0 / _dz(case, n).min()))))
        c, tot, acc = C, 0.0, 0.0
        for a in range(3):
            lo, hi = e.low_high(c, a)
            du = e.diff(ug[a], a)
            c = (c - dt * e.diff(ug[a] * torch.where(ug[a] >= 0, lo, hi), a)) / (1.0 - dt * du)
            acc, tot = acc + c * du, tot + du
        return {"C": (c - dt * acc) / (1.0 - dt * tot)}
    star = _views(_swirl(case, n, seed, centre), vofp.face_shapes(n, bc))
    if kind == "vd":
        g = _gen(seed, 4)
        pn = 0.1 * C + 0.01 * torch.randn(C.shape, dtype=F64, device="cuda", generator=g)
        ph = 2.0 * pn - 0.95 * pn
        dt, rho0 = 1e-3, min(RHO1, RHO2)
        rho = RHO1 * C + RHO2 * (1.0 - C)
        vel = [star[a] - dt * (1.0 / e.face(rho, a) - 1.0 / rho0) * e.grad(ph, a) for a in range(3)]
        vel, p = e.project(vel, None, dt / rho0)
        return {"u": vel, "p": p}
    s, nrm = e.geometry(C, mdot)
    if kind == "extend":
        ue, ug, phi = e.extend(star, s, nrm, mdot)
        return {"ue": ue, "ug": ug, "phi": phi}
    vel, p = e.project(star, s, 1.0)
    ue, ug, _ = e.extend(vel, s, nrm, mdot)
    if kind == "step_host":
        return {"u": vel, "p": p, "ug": ug}
    return {"u": vel, "p": p, "ue": ue, "ug": ug}
