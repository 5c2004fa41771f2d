"""The work that this framework is used for, as cases to be timed and compared.

A case is a problem (geometry, grid, levels), the options of the handle that
solves it, and the call: relaxation sweeps on the finest level (``sweep``), one
multigrid cycle (``vcycle``), a solve (``solve``, ``gmg``), many small solves
at once (``batch``), or a new geometry from nothing to its solution
(``new``).  Geometries and vectors come from the seed; where a solve counts,
the obstacles are the case's (``shapes``), so that it takes as many iterations
for every seed, and the seed gives the flow: force and inflow.

``exact`` discretises the equal-order problems again, by plain torch in 64
bits: element quadrature, Nitsche terms, elimination, local solves, transfers.
"""
import dataclasses
import math

import torch

from paper_2403_11636_gb300 import fc, inputs


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the inner loop of every solve on a 3D pore geometry of the usual size, at the defaults
        dict(name="sweep 3D 64", kind="sweep", geo="porous", dim=3, n=64, m=64, levels=5, spheres=40, prec="fp64",
             cache="inverse", steps=2),
        # the same loop on a large 2D grid, where the vectors no longer fit the L2
        dict(name="sweep 2D 1536", kind="sweep", geo="channel", dim=2, n=1536, m=1536, levels=8, prec="fp64",
             cache="inverse", steps=2),
        # a memory-bound user who keeps factors instead of rows
        dict(name="sweep factors 3D 32", kind="sweep", geo="porous", dim=3, n=32, m=32, levels=4, spheres=40,
             prec="fp64", cache="matrix", steps=2),
        # one preconditioner call of a user's own Krylov loop, float pairs, a grid between the powers of two
        dict(name="cycle pairs 3D 48", kind="vcycle", geo="porous", dim=3, n=48, m=48, levels=4, spheres=40,
             prec="df64", cache="inverse"),
        # the headline solve: flow through 40 spheres to 1e-8
        dict(name="solve 3D 64", kind="solve", geo="porous", dim=3, n=64, m=64, levels=5, spheres=40, prec="fp64",
             cache="inverse", shapes=0),
        # the largest request of a serving stream, float32 rows
        dict(name="solve float 3D 96", kind="solve", geo="porous", dim=3, n=96, m=96, levels=5, spheres=60,
             prec="fp32", cache="inverse", shapes=3),
        # the smallest solve: one obstacle in a 2D channel, where launches and waits count
        dict(name="solve 2D 32", kind="solve", geo="channel", dim=2, n=32, m=32, levels=3, prec="fp64",
             cache="inverse", shapes=1),
        # the published setting: standalone V(6,6) cycles on the long channel, coarse grid of the size table
        dict(name="cycles 2D 1024x256", kind="gmg", geo="replay", dim=2, n=1024, m=256, levels=7, prec="fp64",
             cache="inverse", shapes=1),
        # a parameter study: many uneven 2D problems in one batch
        dict(name="batch 2D of 48", kind="batch", geo="ellipses", dim=2, n=48, shapes=1, levels=0, prec="fp32",
             cache="inverse"),
        # a geometry that is used once: discretisation, patch inverses and the solve
        dict(name="new 3D 32", kind="new", geo="porous", dim=3, n=32, m=32, levels=4, spheres=40, prec="fp64",
             cache="inverse"),
        # quadratic velocities: one cycle of the second element pair in 3D
        dict(name="cycle Q2 3D 16", kind="vcycle", geo="porous", dim=3, n=16, m=16, levels=3, spheres=20,
             prec="fp64", cache="inverse", element="q2"),
        # an octree refined at its obstacle
        dict(name="solve octree 64", kind="solve", geo="duct", dim=3, n=64, m=64, levels=4, prec="fp64",
             cache="inverse", amr=1, shapes=1),
    ]


def _grid(rng, dim, lo, hi, most=18):
    """A size between lo and hi, spread over its logarithm: base * 2^k with k + 1 levels down to `base` cells."""
    size = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    k = max(1, int(math.log2(size / 4.0)) - (rng.randrange(2) if dim == 2 or size < 36 else 0))
    base = max(4, min(9 if dim == 3 else most, round(size / 2 ** k)))
    while base * 2 ** k > hi:
        base -= 1
    return base * 2 ** k, k + 1


def draw(rng):
    what = rng.choice(["sweep3", "sweep2", "factors", "pairs", "solve3", "float3", "solve2", "gmg", "batch", "new",
                       "q2", "octree"])
    if what in ("sweep3", "factors", "pairs", "solve3", "float3", "new"):
        top = {"sweep3": 72, "factors": 36, "pairs": 64, "solve3": 64, "float3": 96, "new": 40}[what]
        n, levels = _grid(rng, 3, 12, top)
        c = dict(geo="porous", dim=3, n=n, m=n, levels=levels, spheres=rng.randint(5, 60),
                 prec="fp64", cache="inverse")
        if what == "sweep3":
            c.update(kind="sweep", steps=rng.randint(1, 4), prec=rng.choice(["fp64", "fp64", "df64", "fp32", "bf16"]))
        elif what == "factors":
            c.update(kind="sweep", steps=rng.randint(1, 2), cache="none" if n <= 20 else "matrix")
        elif what == "pairs":
            c.update(kind="vcycle", prec=rng.choice(["df64", "fp64"]))
        elif what == "solve3":
            c.update(kind="solve", prec=rng.choice(["fp64", "fp64", "df64"]), shapes=rng.randint(4, 99))
        elif what == "float3":
            c.update(kind="solve", prec=rng.choice(["fp32", "fp32", "bf16"]), shapes=rng.randint(4, 99))
        else:
            c.update(kind="new", prec=rng.choice(["fp64", "fp64", "fp32"]))
        return c
    if what == "octree":
        n = rng.choice([32, 40, 48, 56, 64])
        return dict(kind="solve", geo="duct", dim=3, n=n, m=n, levels=4, prec="fp64", cache="inverse",
                    amr=rng.randint(1, 2), shapes=rng.randint(2, 999))
    if what == "q2":
        if rng.random() < 0.5:
            n, levels = _grid(rng, 2, 16, 200)
            return dict(kind="vcycle", geo="channel", dim=2, n=n, m=n, levels=levels, prec="fp64", cache="inverse",
                        element="q2")
        levels = rng.randint(2, 3)
        return dict(kind="vcycle", geo="porous", dim=3, n=4 * 2 ** (levels - 1), m=rng.randint(2, 4) * 2 ** (levels - 1),
                    levels=levels, spheres=rng.randint(2, 30), prec="fp64", cache="inverse", element="q2")
    if what == "batch":
        return dict(kind="batch", geo="ellipses", dim=2, n=rng.randint(4, 48), shapes=rng.randint(2, 999), levels=0,
                    prec=rng.choice(["fp32", "fp32", "fp64"]), cache="inverse")
    if what == "gmg":
        n, levels = _grid(rng, 2, 32, 256, 14)
        return dict(kind="gmg", geo="replay", dim=2, n=4 * n, m=n, levels=levels, prec="fp64", cache="inverse",
                    shapes=rng.randint(2, 99))
    n, levels = _grid(rng, 2, 16, 1536 if what == "sweep2" else 512)
    c = dict(geo=rng.choice(["channel", "ellipse"]), dim=2, n=n, m=n, levels=levels, prec="fp64", cache="inverse")
    if what == "sweep2":
        if rng.random() < 0.5 and n % 2 ** levels == 0:
            c["m"] = n // 2
            c["levels"] -= 1
        c.update(kind="sweep", steps=rng.randint(1, 4), prec=rng.choice(["fp64", "fp64", "df64", "fp32"]))
        if n <= 128:
            c["cache"] = rng.choice(["inverse", "matrix", "none"])
            c["prec"] = c["prec"] if c["cache"] == "inverse" else "fp64"
    else:
        c.update(kind="solve", prec=rng.choice(["fp64", "fp64", "fp32"]), shapes=rng.randint(2, 99))
    return c


def _flow(p, seed):
    """The same geometry under another force and inflow."""
    rng = inputs.SplitMix64(seed)
    return dataclasses.replace(p, force=tuple(f * rng.uniform(0.5, 2.0) for f in p.force), ubar=rng.uniform(0.1, 0.9))


def _problem(c, seed):
    """The problem of a case: what the seed gives (see above), the rest from the case."""
    n, m, lv, flow = c["n"], c["m"], c["levels"], seed
    seed = c.get("shapes", seed)
    if c["geo"] == "porous":
        p = dataclasses.replace(inputs.porous_3d(seed, n=n, nspheres=c["spheres"], nlevels=lv), n=(n, m, m))
    elif c["geo"] == "duct":
        p = inputs.channel_3d(seed, n=n, nlevels=lv)
    elif c["geo"] == "replay":
        p = inputs.channel_replay_2d(seed, nx=n, ny=m, nlevels=lv)
    elif c["geo"] == "channel":
        p = inputs.channel_2d(seed, n=n, nlevels=lv)
    else:
        p = dataclasses.replace(inputs.batch_2d(seed), n=(n, n), nlevels=lv, alpha=1e-8)
    if c["geo"] in ("channel", "ellipse") and m != n:
        p = dataclasses.replace(p, n=(n, m))
    p = _flow(p, flow) if "shapes" in c else p
    return dataclasses.replace(p, amr_uniform=c["amr"]) if "amr" in c else p


def _vector(n, seed, device):
    return torch.as_tensor(inputs.uniform_array(n, 977 * seed + 5, 0.0, 1.0)).to(device)


def prepare(case, seed):
    if case["kind"] == "batch":
        probs = [_flow(inputs.batch_2d(64 * case["shapes"] + k), 64 * seed + k) for k in range(case["n"])]
        batch = fc.Batch([fc.Solver(p, prec=case["prec"]) for p in probs], tile=(16, 256, 8))
        return {"case": case, "batch": batch, "b": batch.rhs()}
    p = _problem(case, seed)
    if case["kind"] == "new":
        return {"case": case, "prob": p}
    s = fc.Solver(p, cache=case["cache"], prec=case["prec"], element=case.get("element", "q1"))
    b = s.rhs()
    # relaxation and cycles meet rough iterates: any start, the problem's own right-hand side
    x = _vector(s.ndof(), seed, b.device)
    return {"case": case, "solver": s, "b": b, "x": x}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "new":
        s = fc.Solver(state["prob"], cache=case["cache"], prec=case["prec"])
        b = s.rhs()
        x, _, _ = s.solve(b)
        s.close()
        return {"rhs": b, "x": x}
    if kind == "batch":
        x, _, _ = state["batch"].solve(state["b"])
        return {"x": x}
    s, b = state["solver"], state["b"]
    if kind == "sweep":
        return {"x": s.smooth(state["x"], b, nsweeps=case["steps"])}
    if kind == "vcycle":
        return {"x": s.vcycle(state["x"], b)}
    if kind == "gmg":
        return {"x": s.gmg_solve(b)[0]}
    return {"x": s.solve(b)[0]}


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    """Operator entries, local rows and vectors, each level and each sweep once.  Rows and entries of nodes away from
    every obstacle are one small block, so those of the cells near a boundary are counted (an estimate by area)."""
    if case["kind"] == "batch":
        one = work(dict(case, kind="solve", geo="ellipse", n=64, m=64, levels=5))
        return {k: case["n"] * v for k, v in one.items()}
    d, n, m, q2 = case["dim"], case["n"], case["m"], case.get("element") == "q2"
    nodes = (n + 1) * (m + 1) * ((m + 1) if d == 3 else 1)
    if "amr" in case:
        nodes //= 20
    slots = (402 if d == 3 else 59) if not q2 else (2214 if d == 3 else 171)
    rows = d + 1 if not q2 else (25 if d == 3 else 9)
    dofs = nodes * rows if q2 else nodes * (d + 1)
    entries = (270 if d == 3 else 63) if not q2 else (2600 if d == 3 else 260)
    cut = 0.65 if d == 3 else min(1.0, 12.0 / min(n, m))
    size = {"fp64": 8, "df64": 8, "fp32": 4, "bf16": 2}[case["prec"]]
    sweep_bytes = 24 * dofs + cut * nodes * (slots * rows * size + 0.8 * entries * size)
    sweep_flops = 2.0 * nodes * (slots * rows + entries)
    if case["cache"] != "inverse":
        sweep_bytes = 24 * dofs + nodes * (39700 if d == 3 else 8000)
        sweep_flops = 2.0 * nodes * ((24000 if d == 3 else 2500) + entries)
    coarser = 1.15 if d == 3 else 1.34
    cycle = {"sweep": case.get("steps", 1), "vcycle": 4 * coarser, "new": 9 * 4 * coarser,
             "solve": (9 if d == 2 else 20) * 4 * coarser, "gmg": 12 * 12 * coarser}[case["kind"]]
    w = {"bytes": cycle * sweep_bytes, "flops": cycle * sweep_flops}
    if case["kind"] == "new":
        w["flops"] += 2.0 * 0.49e6 * cut * nodes * coarser
    return w


# ------------------------------------------------------------------ the same in plain 64-bit torch
def exact(case, seed):
    if case["geo"] == "ellipses" or case.get("element") == "q2" or "amr" in case:
        return None
    p = _problem(case, seed)
    nodes = math.prod(k + 1 for k in p.n)
    kind = case["kind"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if kind in ("sweep", "vcycle"):
        sweeps = case["steps"] if kind == "sweep" else p.nu_pre + p.nu_post
        if nodes * sweeps > (500000 if p.dim == 3 else 6000000):
            return None  # minutes
        fine = _Level(p, p.n, dev)
        x = _vector(nodes * (p.dim + 1), seed, dev)
        if kind == "sweep":
            for _ in range(case["steps"]):
                x = fine.sweep(x, fine.rhs)
            return {"x": x}
        return {"x": _cycle(p, [_Level(p, p.level_n(k), dev) for k in range(1, p.nlevels)] + [fine], x, fine.rhs)}
    if nodes * (p.dim + 1) <= 14000:
        fine = _Level(p, p.n, dev)
        x = fine.direct(fine.rhs)
        return {"rhs": fine.rhs, "x": x} if kind == "new" else {"x": x}
    if kind == "new" and nodes <= 80000:
        return {"rhs": _Level(p, p.n, dev).rhs, "x": None}
    return None


class _Level:
    """A uniform grid: eliminated operator as dense (d+1) x (d+1) blocks to the 3^d neighbours, and its right-hand side."""

    def __init__(self, p, n, dev):
        self.p, self.n, self.d, self.nd, self.dev = p, n, p.dim, p.dim + 1, dev
        self.nn = [k + 1 for k in n]
        self.h = [(b - a) / k for a, b, k in zip(p.lo, p.hi, n)]
        self.nodes = math.prod(self.nn)
        self._assemble()

    def _t(self, *a):
        return torch.tensor(a, dtype=torch.float64, device=self.dev)

    def _phi(self, x, only=None, but=None):
        """The level set at points [..., d]: positive inside an obstacle."""
        out = torch.full(x.shape[:-1], -1.0, dtype=torch.float64, device=self.dev)
        for s, row in enumerate(self.p.shapes):
            if s == but:
                continue
            y = x - self._t(*row[1:1 + self.d])
            if row[0] == 0:
                v = row[4] - y.square().sum(-1).sqrt()
            else:
                u = (row[7] * y[..., 0] + row[8] * y[..., 1]) / row[4]
                w = (row[7] * y[..., 1] - row[8] * y[..., 0]) / row[5]
                v = 1.0 - (u * u + w * w)
            out = v if s == (1 if but == 0 else 0) else torch.maximum(out, v)
        return out

    def _basis(self, x, cell):
        """Values [m, 2^d] and gradients [m, 2^d, d] of the cells' nodal functions at x."""
        low = self._corner(cell)
        h = self._t(*self.h)
        xi = (x - low) / h
        bits = torch.tensor([[(a >> k) & 1 for k in range(self.d)] for a in range(2 ** self.d)], device=self.dev)
        f = torch.where(bits == 1, xi[:, None, :], 1.0 - xi[:, None, :])
        s = torch.where(bits == 1, 1.0, -1.0).to(torch.float64) / h
        grad = []
        for k in range(self.d):
            g = s[:, k].expand(len(x), -1)
            for j in range(self.d):
                g = g * f[:, :, j] if j != k else g
            grad.append(g)
        return f.prod(-1), torch.stack(grad, -1)

    def _index(self, cell, shape):
        out = []
        for k in shape:
            out.append(cell % k)
            cell = cell // k
        return torch.stack(out, -1)

    def _corner(self, cell):
        return self._t(*self.p.lo) + self._index(cell, self.n) * self._t(*self.h)

    def _force(self, x):
        p, f = self.p, torch.zeros_like(x)
        if p.force_kind == 0:
            return f + self._t(*p.force[:self.d])
        f[:, 0] = p.force[0] * torch.sin(math.pi * x[:, 0])
        f[:, 1] = p.force[1] * torch.cos(math.pi * x[:, 1])
        return f

    def _volume_points(self):
        """(point, weight, cell) of the cut-cell rule, in pieces."""
        d, dev = self.d, self.dev
        three = torch.cartesian_prod(*[torch.tensor([0.0, 0.5, 1.0], dtype=torch.float64, device=dev)] * d)
        g = 0.5 / math.sqrt(3.0)
        two = torch.cartesian_prod(*[self._t(0.5 - g, 0.5 + g)] * d)
        child = torch.cartesian_prod(*[self._t(0.0, 0.5)] * d)
        total = math.prod(self.n)
        for first in range(0, total, 20000):
            cell = torch.arange(first, min(total, first + 20000), device=dev)
            low, size = self._corner(cell), self._t(*self.h)
            for depth in range(self.p.qdepth + 1):
                inside = (self._phi(low[:, None, :] + size * three) > 0.0).sum(1)
                cut = (inside > 0) & (inside < len(three)) & (depth < self.p.qdepth)
                done = ~cut
                x = low[done][:, None, :] + size * two
                w = float(size.prod()) / 2 ** d
                yield x.reshape(-1, d), w, cell[done].repeat_interleave(len(two))
                low = (low[cut][:, None, :] + size * child).reshape(-1, d)
                cell = cell[cut].repeat_interleave(len(child))
                size = 0.5 * size
                if not len(low):
                    break

    def _boundary_points(self):
        """(point, normal out of the fluid, weight, cell) on the obstacles."""
        p, d = self.p, self.d
        hmin, fine = min(self.h), 2 ** p.qdepth
        g = 0.5 / math.sqrt(3.0)
        two = self._t(0.5 - g, 0.5 + g)
        for s, row in enumerate(p.shapes):
            c, r = self._t(*row[1:1 + d]), row[4]
            if d == 2:
                big = max(row[4], row[5]) if row[0] else r
                count = max(64, 8 * math.ceil(2.0 * math.pi * big / hmin) * fine)
                dt = 2.0 * math.pi / count
                t = (dt * (torch.arange(count, dtype=torch.float64, device=self.dev)[:, None] + two)).reshape(-1)
                a, b, cr, sr = (r, row[5], row[7], row[8]) if row[0] else (r, r, 1.0, 0.0)
                ct, st = torch.cos(t), torch.sin(t)
                x = c + torch.stack([cr * a * ct - sr * b * st, sr * a * ct + cr * b * st], -1)
                normal = torch.stack([cr * b * ct - sr * a * st, sr * b * ct + cr * a * st], -1)
                normal = -normal / normal.square().sum(-1, keepdim=True).sqrt()
                w = 0.5 * dt * ((a * st).square() + (b * ct).square()).sqrt()
            else:
                count = max(8, math.ceil(2.0 * r / hmin) * fine)
                turn = max(16, 2 * math.ceil(2.0 * math.pi * r / hmin) * fine)
                dm, df = 2.0 / count, 2.0 * math.pi / turn
                mu = (-1.0 + dm * (torch.arange(count, dtype=torch.float64, device=self.dev)[:, None] + two)).reshape(-1, 1)
                ph = df * (torch.arange(turn, dtype=torch.float64, device=self.dev) + 0.5)
                st = (1.0 - mu * mu).sqrt()
                e = torch.stack([st * torch.cos(ph), st * torch.sin(ph), mu.expand(-1, turn)], -1).reshape(-1, 3)
                x, normal = c + r * e, -e
                w = torch.full((len(e),), r * r * 0.5 * dm * df, dtype=torch.float64, device=self.dev)
            lo, hi = self._t(*p.lo), self._t(*p.hi)
            keep = ((x >= lo) & (x <= hi)).all(-1)
            if len(p.shapes) > 1:
                keep &= ~(self._phi(x, but=s) > 0.0)
            x, normal, w = x[keep], normal[keep], w[keep]
            i = torch.floor((x - lo) / self._t(*self.h)).long()
            i = torch.minimum(i.clamp(min=0), torch.tensor(self.n, device=self.dev) - 1)
            cell = i[:, -1]
            for k in range(d - 2, -1, -1):
                cell = cell * self.n[k] + i[:, k]
            for first in range(0, len(x), 400000):
                at = slice(first, first + 400000)
                yield x[at], normal[at], w[at], cell[at]

    def _assemble(self):
        p, d, nd, q, dev = self.p, self.d, self.nd, 2 ** self.d, self.dev
        cells = math.prod(self.n)
        zero = lambda *s: torch.zeros(*s, dtype=torch.float64, device=dev)  # noqa: E731
        A, B, F = zero(cells, q, q), zero(cells, d, q, q), zero(cells, d, q)
        for x, w, cell in self._volume_points():
            val, grad = self._basis(x, cell)
            al = w * torch.where(self._phi(x) > 0.0, p.alpha, 1.0).to(torch.float64)
            A.index_add_(0, cell, torch.einsum("mak,mbk,m->mab", grad, grad, p.eta * al))
            B.index_add_(0, cell, -torch.einsum("mac,mb,m->mcab", grad, val, al))
            F.index_add_(0, cell, torch.einsum("mc,ma,m->mca", self._force(x), val, al))
        lam = p.beta * p.eta / min(self.h)
        for x, normal, w, cell in self._boundary_points():
            val, grad = self._basis(x, cell)
            dn = torch.einsum("mk,mak->ma", normal, grad)
            t = torch.einsum("ma,mb->mab", val, dn)
            A.index_add_(0, cell, (lam * torch.einsum("ma,mb->mab", val, val) - p.eta * (t + t.mT)) * w[:, None, None])
            B.index_add_(0, cell, torch.einsum("ma,mc,mb,m->mcab", val, normal, val, w))
        one = self._t(1.0 / 3, 1.0 / 6, 1.0 / 6, 1.0 / 3).reshape(2, 2)
        mass = torch.ones(1, 1, dtype=torch.float64, device=dev)
        for k in range(d):
            mass = torch.kron(one * self.h[k], mass)
        vol = math.prod(self.h)
        C = -(mass - vol / q ** 2) / p.eta
        E = zero(cells, q, nd, q, nd)
        for c in range(d):
            E[:, :, c, :, c] = A
            E[:, :, c, :, d] = B[:, c]
            E[:, :, d, :, c] = B[:, c].mT
        E[:, :, d, :, d] = C
        del A, B
        # nodes of cells, and the neighbour slot of one local node seen from another
        ic = self._index(torch.arange(cells, device=dev), self.n)
        st, f = zero(self.nodes, 3 ** d, nd, nd), zero(self.nodes, nd)
        bit = [[(a >> k) & 1 for k in range(d)] for a in range(q)]
        for a in range(q):
            node = self._node(ic + torch.tensor(bit[a], device=dev))
            f[:, :d].index_add_(0, node, F[:, :, a])
            for b in range(q):
                slot = sum((bit[b][k] - bit[a][k] + 1) * 3 ** k for k in range(d))
                st[:, slot].index_add_(0, node, E[:, a, :, b, :])
        del E
        # strong data on the box faces, eliminated symmetrically
        i = self._index(torch.arange(self.nodes, device=dev), self.nn)
        wall = torch.zeros(self.nodes, dtype=torch.bool, device=dev)
        for k in range(1, d):
            wall |= (i[:, k] == 0) | (i[:, k] == self.n[k])
        value = zero(self.nodes, nd)
        if p.preset == 0:
            flow = (i[:, 0] == 0) & ~wall
            prof = torch.full((self.nodes,), p.ubar, dtype=torch.float64, device=dev)
            for k in range(1, d):
                s = i[:, k].double() / self.n[k]
                prof = prof * 4.0 * s * (1.0 - s)
            value[:, 0] = torch.where(flow, prof, 0.0)
            wall = wall | flow
        self.fixed = torch.zeros(self.nodes, nd, dtype=torch.bool, device=dev)
        self.fixed[:, :d] = wall[:, None]
        self.i, self.st = i, st
        self.nb, self.has = self._around(torch.arange(self.nodes, device=dev), 1)
        xf = self._pad(value)[self.nb]
        f = f - torch.einsum("nsab,nsb->na", st, xf)
        out = self._pad(self.fixed)[self.nb]
        st.masked_fill_(out[:, :, None, :], 0.0)
        st.masked_fill_(self.fixed[:, None, :, None], 0.0)
        st[:, (3 ** d) // 2] += torch.diag_embed(self.fixed.double())
        self.rhs = torch.where(self.fixed, value, f).reshape(-1)

    def _node(self, i):
        n = i[..., -1]
        for k in range(self.d - 2, -1, -1):
            n = n * self.nn[k] + i[..., k]
        return n

    def _around(self, node, r):
        """The (2r+1)^d nodes around each (x fastest; self.nodes where the grid ends), and which there are."""
        o = torch.arange(-r, r + 1, device=self.dev)
        o = torch.cartesian_prod(*[o] * self.d).flip(-1)
        j = self.i[node][:, None, :] + o
        ok = ((j >= 0) & (j < torch.tensor(self.nn, device=self.dev))).all(-1)
        return torch.where(ok, self._node(j), self.nodes), ok

    def _pad(self, v):
        return torch.cat([v, torch.zeros_like(v[:1])])

    def residual(self, x, b):
        y = x.reshape(-1, self.nd)
        return (b.reshape(-1, self.nd) - torch.einsum("nsab,nsb->na", self.st, self._pad(y)[self.nb])).reshape(-1)

    def sweep(self, x, b):
        """x after one restricted additive relaxation: every node's own unknowns of its patch's exact solution."""
        d, nd = self.d, self.nd
        r = self._pad(self.residual(x, b).reshape(-1, nd))
        fixed = self._pad(self.fixed)
        # entries of patch matrices: velocity nodes of the 5^d box, pressures of the 3^d box
        box = torch.cartesian_prod(*[torch.arange(-2, 3, device=self.dev)] * d).flip(-1)
        small = (box.abs() <= 1).all(-1).nonzero()[:, 0]
        off = box[None, :, :] - box[:, None, :]
        near = (off.abs() <= 1).all(-1)
        slot = sum((off[..., k].clamp(-1, 1) + 1) * 3 ** k for k in range(d))
        mid, own = len(box) // 2, len(small) // 2
        st = self._pad(self.st)
        y = torch.zeros_like(r)
        step = 3000 if d == 3 else 30000
        for first in range(0, self.nodes, step):
            at = torch.arange(first, min(self.nodes, first + step), device=self.dev)
            node, ok = self._around(at, 2)
            free = ok & ~fixed[node][..., 0]
            there = ok[:, small]
            sb = st[node]
            pick = slot.expand(len(at), -1, -1)
            entry = lambda a, b: torch.gather(sb[..., a, b], 2, pick) * near  # noqa: E731
            eye = torch.eye(len(box), dtype=torch.float64, device=self.dev)
            K = entry(0, 0) * (free[:, :, None] & free[:, None, :]) + eye * ~free[:, None, :]
            B = [entry(c, d)[:, :, small] * (free[:, :, None] & there[:, None, :]) for c in range(d)]
            C = entry(d, d)[:, small][:, :, small] * (there[:, :, None] & there[:, None, :])
            C = C + torch.eye(len(small), dtype=torch.float64, device=self.dev) * ~there[:, None, :]
            du = K.diagonal(dim1=1, dim2=2).abs().rsqrt()[:, :, None]
            dp = C.diagonal(dim1=1, dim2=2).abs().rsqrt()[:, :, None]
            K, C = K * du * du.mT, C * dp * dp.mT
            B = [v * du * dp.mT for v in B]
            ru = [(r[node][..., c] * free)[:, :, None] * du for c in range(d)]
            rp = (r[node][:, small, d] * there)[:, :, None] * dp
            lu = torch.linalg.lu_factor(K)
            w = torch.linalg.lu_solve(*lu, torch.cat(B + ru, -1))
            q = len(small)
            S, g = C, rp
            for c in range(d):
                S = S - B[c].mT @ w[..., c * q:(c + 1) * q]
                g = g - B[c].mT @ w[..., d * q + c:d * q + c + 1]
            z = torch.linalg.solve(S, g)
            y[at, d] = (z * dp)[:, own, 0]
            for c in range(d):
                u = w[:, mid, d * q + c] - (w[:, mid, c * q:(c + 1) * q] * z[..., 0]).sum(-1)
                y[at, c] = u * du[:, mid, 0]
        r, y = r[:-1], y[:-1]
        return (x.reshape(-1, nd) + torch.where(self.fixed, r, self.p.omega * y)).reshape(-1)

    def direct(self, b):
        """The solution, by a dense factorisation of the scaled operator."""
        nd, size = self.nd, (self.nodes + 1) * self.nd
        L = torch.zeros(size, size, dtype=torch.float64, device=self.dev)
        row = torch.arange(self.nodes, device=self.dev)[:, None, None, None] * nd + torch.arange(nd, device=self.dev)[:, None]
        col = self.nb[:, :, None, None] * nd + torch.arange(nd, device=self.dev)
        L.index_put_((row.expand_as(self.st), col.expand_as(self.st)), self.st, accumulate=True)
        L = L[:-nd, :-nd]
        s = L.diagonal().abs().rsqrt()
        return s * torch.linalg.solve(L * s[:, None] * s, (s * b)[:, None])[:, 0]


def _weights(nc, dev):
    """Linear interpolation from nc + 1 to 2 nc + 1 nodes."""
    w = torch.zeros(2 * nc + 1, nc + 1, dtype=torch.float64, device=dev)
    for i in range(2 * nc + 1):
        w[i, i // 2] += 0.5
        w[i, (i + 1) // 2] += 0.5
    return w


def _transfer(coarse, v, up):
    d, nd = coarse.d, coarse.nd
    n = [2 * k + 1 for k in coarse.n] if not up else coarse.nn
    v = v.reshape(*reversed(n), nd)
    for k in range(d):
        w = _weights(coarse.n[k], coarse.dev)
        ax = d - 1 - k
        v = torch.tensordot(w if up else w.mT, v, dims=([1], [ax])).movedim(0, ax)
    return v.reshape(-1, nd)


def _cycle(p, levels, x, b):
    fine = levels[-1]
    if len(levels) == 1:
        return fine.direct(b)
    for _ in range(p.nu_pre):
        x = fine.sweep(x, b)
    coarse = levels[-2]
    bc = torch.where(coarse.fixed, 0.0, _transfer(coarse, fine.residual(x, b), False)).reshape(-1)
    e = _cycle(p, levels[:-1], torch.zeros_like(bc), bc)
    x = x + torch.where(fine.fixed, 0.0, _transfer(coarse, e, True)).reshape(-1)
    for _ in range(p.nu_post):
        x = fine.sweep(x, b)
    return x
