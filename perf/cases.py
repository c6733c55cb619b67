"""The workloads by which this library's speed is judged.

A case is one call sequence of a user's program: install a checkpoint in a handle (or a batch),
advance it by a number of explicit steps (Poisson solve, fields, time step, fluxes, update) and
take the checkpoint back, through the public Python binding and pinned host buffers.  Sizes,
voltages, densities and closures are those of `workloads.py`, of the tests and of `bench.py`;
`draw` spreads them over the ranges between the smallest test meshes and 2,000,000 nodes.

`exact` advances the same problem in plain 64-bit torch: textbook assembly by scatter-adds over
the cells and solves to round-off (dense LU on small meshes, Jacobi-preconditioned Krylov
iteration on larger ones), none of this library's code.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2201_01291_gb300 import avip, workloads

MAX_BATCH = 16
DENSE = 12000       # nodes up to which `exact` factorises the whole matrix


# --------------------------------------------------------------------------- the cases
def listed():
    def case(name, family, nx, ny, steps, precision="fp64", scheme="llw"):
        return {"name": name, "family": family, "nx": nx, "ny": ny, "steps": steps, "precision": precision,
                "scheme": scheme}

    return [
        # the smallest call: one step of a 17 x 17 test mesh, as a program that owns the time loop makes it
        case("step_plates_17x17", "plates", 17, 17, 1),
        # parallel plates, 65 x 65 nodes, 100 steps: the plain FP64 configuration and its mixed-precision form
        case("plates_65x65", "plates", 65, 65, 100),
        case("plates_65x65_mixed", "plates", 65, 65, 100, precision="mixed"),
        # pin-plane streamer on a coarse mesh, as a parameter scan or a convergence study runs it
        case("pin_plane_151x301", "pin_plane", 151, 301, 20),
        # the pin-plane streamer of the benchmark, FP64 and mixed precision
        case("pin_plane_500x1000", "pin_plane", 500, 1000, 20),
        case("pin_plane_500x1000_mixed", "pin_plane", 500, 1000, 20, precision="mixed"),
        # the largest single mesh: 2,000,000 nodes, the upper end of the size sweep
        case("pin_plane_1000x2000", "pin_plane", 1000, 2000, 8),
        # three-species air chemistry under a voltage ramp
        case("three_species_401x399", "three_species", 401, 399, 20),
        # triangles and quadrangles together, Scharfetter-Gummel fluxes
        case("hybrid_251x501_sg", "hybrid", 251, 501, 20, scheme="sg"),
        # axisymmetric streamer gap (non-symmetric matrix), and a coarser one with photoionisation
        case("axisym_701x701", "axisym", 701, 701, 12),
        case("axisym_photo_251x251", "axisym_photo", 251, 251, 8),
        # uneven independent instances advanced together, in the precision batches are run in
        {"name": "batch_16_mixed", "family": "batch", "count": 16, "t_min": 2000, "t_max": 200000, "steps": 8,
         "precision": "mixed", "scheme": "llw"},
    ]


def draw(rng):
    """One more case: family, size (log-uniform in the nodes), aspect, precision and scheme."""
    family = rng.choice(["plates", "plates", "pin_plane", "pin_plane", "pin_plane", "three_species", "hybrid",
                         "axisym", "axisym_photo", "batch"])
    if family == "batch":
        t_min = rng.randint(2000, 6000)
        return {"family": family, "count": rng.randint(5, MAX_BATCH), "t_min": t_min,
                "t_max": int(t_min * math.exp(rng.uniform(math.log(4.0), math.log(30.0)))),
                "steps": rng.randint(4, 8), "precision": rng.choice(["fp64", "mixed"]), "scheme": "llw"}
    lo, hi, aspect = {"plates": (120, 9000, 1.0), "pin_plane": (9000, 1500000, 2.0),
                      "three_species": (8000, 400000, 1.0), "hybrid": (5000, 300000, 2.0),
                      "axisym": (2500, 450000, 1.0), "axisym_photo": (2500, 120000, 1.0)}[family]
    nodes = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    shape = aspect * rng.uniform(0.8, 1.25)
    nx = max(9, int(round(math.sqrt(nodes / shape))))
    ny = max(9, int(round(nodes / nx)))
    if family == "plates":
        steps = rng.randint(1, 100)
    elif family == "axisym_photo":
        steps = rng.randint(4, 8)
    else:
        steps = rng.randint(4, 6) if nodes > 500000 else rng.randint(6, 16)
    mixed = family in ("plates", "pin_plane") and rng.random() < 0.35
    return {"family": family, "nx": nx, "ny": ny, "steps": steps, "precision": "mixed" if mixed else "fp64",
            "scheme": "sg" if rng.random() < 0.2 and not mixed else "llw"}


def problems(case, seed):
    """The workload descriptions of a case (one, or a batch's instances); the seed moves every node."""
    w, family = workloads, case["family"]
    if family == "batch":
        out = []
        for k, q in enumerate(w.random_instances(case["count"], 3, t_min=case["t_min"], t_max=case["t_max"])):
            m, ns = q.meta, len(q.species)  # sizes, voltage and species are the case's
            out.append(w.plates_problem(m["nx"], m["ny"], m["Lx"], m["Ly"], m["voltage"], seed * 1009 + k,
                                        field_dependent=True, source=q.source.model, n_species=ns))
        return out
    nx, ny, scheme = case["nx"], case["ny"], w.FLUX_SG if case["scheme"] == "sg" else w.FLUX_LLW
    # axisymmetric solves run at the tolerance of their tests: near the axis the densities carry
    # several hundred times the residual
    opts = w.Opts(scheme=scheme, rtol=1e-13 if family.startswith("axisym") else 1e-12)
    streamer = dict(field_dependent=True, source=w.SRC_TOWNSEND, opts=opts)
    if family == "plates":
        p = w.plates_problem(nx, ny, 1e-2, 1e-2, 5e3, seed, opts=opts)
    elif family == "pin_plane":
        p = w.plates_problem(nx, ny, 1e-2, 2e-2, 2e4, seed, needle_len=2e-3, **streamer)
    elif family == "three_species":
        p = w.morrow_lowke_problem(nx, ny, 5e-3, 5e-3, 5e3, seed, needle_len=1e-3, opts=opts)
    elif family == "hybrid":
        p = w.hybrid_plates_problem(nx, ny, 1e-2, 2e-2, 2e4, seed, quad_fraction=0.5, needle_len=2e-3, **streamer)
    else:  # axisym, axisym_photo
        photo = family == "axisym_photo"
        p = w.axisym_problem(nx, ny, 1.25e-2, 1.25e-2, 18750.0, seed, n_peak=5e18, n_back=1e9 if photo else 1e13,
                             sigma=4e-4, x0=1e-2, **streamer)
        p.photo = w.photo_air() if photo else None
    return [p]


# --------------------------------------------------------------------------- one pass
class Run:
    """The handle (or batch) a program keeps, the checkpoint it starts from and the buffer it ends in."""

    def __init__(self, case, seed):
        ps = problems(case, seed)
        precision = avip.PREC_MIXED if case["precision"] == "mixed" else avip.PREC_FP64
        self.meshes = [avip.Mesh(p, precision=precision) for p in ps]
        self.shapes = [(len(p.species), p.n_nodes) for p in ps]
        self.steps = case["steps"]
        self.handle = avip.Batch(self.meshes) if case["family"] == "batch" else self.meshes[0]
        size = sum((ns + 4) * n + 2 for ns, n in self.shapes)
        self.start = torch.empty(size, dtype=torch.float64, pin_memory=True).numpy()
        self.out = torch.empty(size, dtype=torch.float64, pin_memory=True).numpy()
        self.handle.state(out=self.start)

    def __del__(self):
        if isinstance(getattr(self, "handle", None), avip.Batch):
            self.handle.close()  # before the handles it advances
        for m in getattr(self, "meshes", []):
            m.close()


def prepare(case, seed):
    return Run(case, seed)


def run(state):
    state.handle.set_state(state.start)
    if state.steps == 1 and isinstance(state.handle, avip.Mesh):
        state.handle.step()
    else:
        state.handle.run(state.steps)
    flat = state.handle.state(out=state.out)
    outs, at = [], 0
    for ns, n in state.shapes:
        part = flat[at:at + (ns + 4) * n + 2]
        outs.append(fields(part, ns, n, state.steps))
        at += part.size
    return outs


def fields(flat, ns, n, steps):
    """A checkpoint's densities, potential, time and the earlier potentials of the solver's predictor."""
    k = ns * n
    out = {"density": flat[:k].reshape(ns, n), "phi": flat[k:k + n], "t": flat[k + n:k + n + 1]}
    if steps > 1:
        out["earlier_phi"] = flat[k + n + 1:k + n + 1 + 3 * n].reshape(3, n)[:min(3, steps - 1)]
    return out


def sizes(case):
    """(nodes, cells, edges, stored matrix entries, species) summed over a case's meshes."""
    if case["family"] == "batch":
        mean = (case["t_max"] - case["t_min"]) / math.log(case["t_max"] / case["t_min"])
        cells = case["count"] * mean
        n, ns = 0.5 * cells + case["count"], 2.5
    else:
        nx, ny = case["nx"], case["ny"]
        n, cells = nx * ny, 2 * (nx - 1) * (ny - 1)
        cells *= 0.75 if case["family"] == "hybrid" else 1.0
        ns = 3 if case["family"] == "three_species" else 2
    edges = n + cells
    return n, cells, edges, n + 2 * edges, ns


def work(case):
    """Per step: the matrix and the edge geometry read once, the densities read and written, the
    potential written, the cells read; the checkpoint in and out once per pass."""
    n, cells, edges, nnz, ns = sizes(case)
    solves = 4 if case["family"] == "axisym_photo" else 1
    step = 12 * nnz * solves + 24 * edges + 16 * cells + n * (16 * ns + 8 * solves + 32)
    flops = 2 * nnz * (solves + 1 + ns) + 40 * ns * edges + 20 * ns * cells + 60 * n
    return {"bytes": case["steps"] * step + 16 * (ns + 4) * n, "flops": case["steps"] * flops}


# --------------------------------------------------------------------------- 64-bit values
def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    outs = []
    for p in problems(case, seed):
        density, phis, t = Plain(p, device).advance(case["steps"])
        out = {"density": torch.stack(density), "phi": phis[-1], "t": t.reshape(1)}
        if case["steps"] > 1:
            out["earlier_phi"] = torch.stack(phis[-2:-5:-1])
        outs.append(out)
    return outs


class Plain:
    """The explicit step on one mesh in 64-bit torch: cell loops and scatter-adds."""

    def __init__(self, p, device):
        self.p, self.dev = p, device
        self.xy = self.put(p.xy)
        self.n = p.n_nodes
        groups = [c for c in (p.tris, p.quads) if c is not None and len(c)]
        self.cells = [self.put(c, torch.int64).reshape(len(c), -1) for c in groups]
        self.fixed = self.put(p.node_bc, torch.int64) == 1
        self.phi_d = torch.where(self.fixed, self.put(p.phi_D), 0.0)
        self.geometry()
        self.operators()

    def put(self, a, dtype=torch.float64):
        return torch.as_tensor(np.ascontiguousarray(a), device=self.dev).to(dtype)

    def scatter(self, index, values, size=None):
        out = torch.zeros((size or self.n,) + values.shape[1:], dtype=values.dtype, device=self.dev)
        return out.index_add_(0, index, values)

    def geometry(self):
        """Areas, nodal normals, dual volumes, and the dual faces of edges and boundary nodes."""
        axi = self.p.axisymmetric
        self.area, self.normal, self.short = [], [], []
        self.planar = torch.zeros(self.n, dtype=torch.float64, device=self.dev)
        volume = torch.zeros_like(self.planar)
        tail, head, dual, face, weight = [], [], [], [], []
        for c in self.cells:
            nv = c.shape[1]
            x = self.xy[c]                                             # (cells, nv, 2), counter-clockwise
            nxt = x.roll(-1, 1)
            a = 0.5 * (x[..., 0] * nxt[..., 1] - nxt[..., 0] * x[..., 1]).sum(1)
            side = nxt - x
            out = torch.stack([side[..., 1], -side[..., 0]], -1)       # outward face normals
            s = -(out + out.roll(1, 1))                                # nodal normals
            self.area.append(a)
            self.normal.append(s)
            self.short.append(side.norm(dim=-1).min(1).values)
            share = (a / nv)[:, None].expand(-1, nv)
            self.planar.index_add_(0, c.reshape(-1), share.reshape(-1))
            r = x[..., 1]
            rev = a[:, None] * (15.0 * r + 7.0 * r.sum(1, keepdim=True)) / 108.0 if axi else share
            volume.index_add_(0, c.reshape(-1), rev.reshape(-1))
            mid, centre = 0.5 * (x + nxt), x.mean(1, keepdim=True)
            d = centre - mid
            d = torch.stack([d[..., 1], -d[..., 0]], -1)
            d = d * torch.sign((d * side).sum(-1, keepdim=True))
            if axi:
                d = d * (0.5 * (mid[..., 1] + centre[..., 1]))[..., None]
            tail.append(c.reshape(-1))
            head.append(c.roll(-1, 1).reshape(-1))
            dual.append(d.reshape(-1, 2))
            face.append(0.5 * out.reshape(-1, 2))
            rn = nxt[..., 1]
            weight.append(torch.stack([(3 * r + rn) / 4, (r + 3 * rn) / 4], -1).reshape(-1, 2))
        tail, head, dual, face, weight = (torch.cat(v) for v in (tail, head, dual, face, weight))
        if not axi:
            weight = torch.ones_like(weight)
        self.volume = volume
        swap = tail > head
        key = torch.minimum(tail, head) * self.n + torch.maximum(tail, head)
        key, edge, count = torch.unique(key, return_inverse=True, return_counts=True)
        self.lo, self.hi = key // self.n, key % self.n
        self.dual = self.scatter(edge, torch.where(swap[:, None], -dual, dual), key.numel())
        rim = count[edge] == 1
        self.rim = (self.scatter(tail[rim], face[rim] * weight[rim, :1])
                    + self.scatter(head[rim], face[rim] * weight[rim, 1:]))

    def operators(self):
        """The Poisson matrix over all vertex pairs of a cell, with the fixed nodes eliminated."""
        rows, cols, vals = [], [], []
        for c, a, s in zip(self.cells, self.area, self.normal):
            nv = c.shape[1]
            if self.p.axisymmetric:
                r = self.xy[c][..., 1]
                rt, tot = r.mean(1, keepdim=True), r.sum(1, keepdim=True)
                own = 4 * rt + r + tot                                 # 4 r_tau + 2 r_k + r_j + r_l
                w = torch.zeros_like(s)
                for k in range(3):
                    j, l = (k + 1) % 3, (k + 2) % 3
                    w[:, k] = (own[:, k, None] * s[:, k] - (2 * rt + r[:, k, None] + r[:, j, None]) * s[:, j]
                               - (2 * rt + r[:, k, None] + r[:, l, None]) * s[:, l]) / 24.0
                pair = torch.einsum("cid,cjd->cij", w, s) / (2.0 * a)[:, None, None]
            else:
                pair = torch.einsum("cid,cjd->cij", s, s) / (4.0 * a)[:, None, None]
            rows.append(c[:, :, None].expand(-1, nv, nv).reshape(-1))
            cols.append(c[:, None, :].expand(-1, nv, nv).reshape(-1))
            vals.append(pair.reshape(-1))
        rows, cols, vals = torch.cat(rows), torch.cat(cols), torch.cat(vals)
        key, at = torch.unique(rows * self.n + cols, return_inverse=True)
        vals = self.scatter(at, vals, key.numel())
        rows, cols = key // self.n, key % self.n
        self.row, self.col, self.val = rows, cols, vals
        fd = ~self.fixed[rows] & self.fixed[cols]
        self.lift = -self.scatter(rows[fd], vals[fd] * self.phi_d[cols[fd]])
        terms = self.p.photo.kappa if self.p.photo is not None else []
        self.systems = [self.system(0.0)] + [self.system(k * k) for k in terms]

    def system(self, shift):
        """Unit rows for the fixed nodes, K + shift V for the others, scaled to a unit diagonal."""
        free = ~self.fixed[self.row] & ~self.fixed[self.col]
        same = self.row == self.col
        val = torch.where(same, self.val + shift * self.volume[self.row], self.val)
        val = torch.where(free, val, torch.where(same, 1.0, 0.0))
        diag = self.scatter(self.row[same], val[same])
        root = diag.rsqrt()
        keep = val != 0
        r, c = self.row[keep], self.col[keep]
        start = torch.zeros(self.n + 1, dtype=torch.int64, device=self.dev)
        start[1:] = torch.cumsum(torch.bincount(r, minlength=self.n), 0)
        v = val[keep] * root[r] * root[c]
        if self.n <= DENSE:
            dense = torch.zeros(self.n, self.n, dtype=torch.float64, device=self.dev)
            dense[r, c] = v
            return dense, root, torch.linalg.lu_factor(dense)
        m = torch.sparse_csr_tensor(start, c, v, (self.n, self.n))
        return m, root, None

    def solve(self, system, b, guess):
        """The scaled system to round-off: LU with one refinement, or CG (BiCGStab where it is not symmetric)."""
        m, root, lu = system
        b, x = b * root, guess / root
        if lu is not None:
            x = torch.linalg.lu_solve(*lu, b[:, None])[:, 0]
            return root * (x + torch.linalg.lu_solve(*lu, (b - m @ x)[:, None])[:, 0])
        scale = float(b.norm())
        if scale == 0.0:
            return torch.zeros_like(b)
        best, kept = math.inf, x
        for _ in range(6):  # restarts from the true residual until it stops falling
            r = b - m @ x
            now = float(r.norm())
            if now < best:
                kept, gain, best = x, best / max(now, 1e-300), now
            if best <= 2e-15 * scale or now > best or gain < 3.0:
                break
            x = (self.bicgstab if self.p.axisymmetric else self.cg)(m, x.clone(), r, 1e-15 * scale)
        return kept * root

    @staticmethod
    def cg(m, x, r, stop):
        p, rr = r.clone(), r @ r
        for it in range(1, 20001):
            q = m @ p
            al = rr / (p @ q)
            x += al * p
            r -= al * q
            new = r @ r
            p.mul_(new / rr).add_(r)
            rr = new
            if it % 40 == 0 and not float(rr) > stop * stop:
                break
        return x

    @staticmethod
    def bicgstab(m, x, r, stop):
        shadow, p, rho = r.clone(), r.clone(), r @ r
        for it in range(1, 4001):
            v = m @ p
            al = rho / (shadow @ v)
            s = r - al * v
            t = m @ s
            om = (t @ s) / (t @ t)
            step = al * p + om * s
            x += step
            r = s - om * t
            new = shadow @ r
            p = r + (new / rho) * (al / om) * (p - om * v)
            rho = new
            if it % 20 == 0 or it < 4:
                size = float(r.norm())
                if not math.isfinite(size):
                    return x - step
                if size <= stop:
                    break
        return x

    def gradient(self, u):
        g = torch.zeros(self.n, 2, dtype=torch.float64, device=self.dev)
        for c, s in zip(self.cells, self.normal):
            cell = -(u[c][..., None] * s).sum(1) / (2.0 * c.shape[1])  # area/nv times the cell gradient
            g.index_add_(0, c.reshape(-1), cell[:, None].expand(-1, c.shape[1], -1).reshape(-1, 2))
        return g / self.planar[:, None]

    def sources(self, n, size, mu, guesses):
        src, p = self.p.source, self.p
        out = [torch.zeros_like(size) for _ in n]
        if src.model == workloads.SRC_NONE:
            return out
        e, pos, neg = src.idx
        rate = lambda a, b: torch.where(size > 0, a * torch.exp(-b / size), 0.0) * mu[e] * size * n[e]  # noqa: E731
        ion = rate(src.params[0], src.params[1])
        out[e], out[pos] = out[e] + ion, out[pos] + ion
        if src.model == workloads.SRC_TOWNSEND_ATTACH:
            out[e], out[neg] = out[e] - src.params[2] * n[e], out[neg] + src.params[2] * n[e]
        elif src.model == workloads.SRC_MORROW_LOWKE:
            att = rate(src.params[2], src.params[3])
            ep, np_ = src.params[4] * n[e] * n[pos], src.params[4] * n[neg] * n[pos]
            out[e], out[pos], out[neg] = out[e] - att - ep, out[pos] - ep - np_, out[neg] + att - np_
        if p.photo is not None:
            for j, a in enumerate(p.photo.a):
                b = torch.where(self.fixed, 0.0, a * self.volume * p.photo.c * ion)
                guesses[j] = self.solve(self.systems[1 + j], b, guesses[j])
                out[e], out[pos] = out[e] + guesses[j], out[pos] + guesses[j]
        return out

    def time_step(self, n, mu, vel, s_e):
        o, limits = self.p.opts, []
        for c, dx in zip(self.cells, self.short):
            sigma = torch.zeros_like(dx)
            for k, sp in enumerate(self.p.species):
                speed = vel[k][c].mean(1).norm(dim=-1)
                limits.append((o.cfl * dx / speed).min())
                if sp.D > 0:
                    limits.append((o.fourier * dx * dx / sp.D).min())
                sigma += (sp.charge * workloads.E_CHARGE * (n[k] * mu[k])[c].mean(1)).abs()
            limits.append((o.a_diel * workloads.EPS0 / sigma).min())
        if self.p.source.model != workloads.SRC_NONE:
            n_e = n[self.p.source.idx[0]]
            limits.append(torch.where(s_e != 0, o.a_chem * n_e.abs() / s_e.abs(), math.inf).min())
        return torch.stack(limits).min()

    def flux(self, u, grad, vel, d, dt):
        """Flux from lo to hi through every dual face."""
        lo, hi, s = self.lo, self.hi, self.dual
        v, g = 0.5 * (vel[lo] + vel[hi]), 0.5 * (grad[lo] + grad[hi])
        dx = self.xy[hi] - self.xy[lo]
        if self.p.opts.scheme == workloads.FLUX_SG:
            h = dx.norm(dim=-1)
            e = dx / h[:, None]
            along = (s * e).sum(-1)
            across = s - along[:, None] * e
            vt = (v * e).sum(-1)
            if d > 0:
                a = h * vt / d
                bern = lambda z: torch.where(z == 0, 1.0, z / torch.expm1(z))  # noqa: E731
                f = d * along / h * (bern(-a) * u[lo] - bern(a) * u[hi])
            else:
                f = along * (vt.clamp(min=0) * u[lo] + vt.clamp(max=0) * u[hi])
            return f + (v * across).sum(-1) * 0.5 * (u[lo] + u[hi]) - d * (g * across).sum(-1)
        through = (v * s).sum(-1)
        first = through >= 0
        up, down = torch.where(first, lo, hi), torch.where(first, hi, lo)
        delta = u[down] - u[up]
        ahead = 2.0 * (grad[up] * torch.where(first[:, None], dx, -dx)).sum(-1) - delta
        psi = torch.where(delta != 0, (ahead / delta).clamp(0.0, 1.0), 0.0)  # min-mod, the default limiter
        wave = 0.5 * delta - 0.5 * dt * (g * v).sum(-1)
        return (u[up] + wave * psi) * through - d * (g * s).sum(-1)

    def advance(self, steps):
        p, phi = self.p, torch.zeros(self.n, dtype=torch.float64, device=self.dev)
        n = [self.put(sp.n0) for sp in p.species]
        t = torch.zeros((), dtype=torch.float64, device=self.dev)
        phis, guesses = [], [torch.zeros_like(phi) for _ in self.systems[1:]]
        for _ in range(steps):
            gain = (t / p.opts.v_rise).clamp(max=1.0) if p.opts.v_rise > 0 else 1.0
            rho = sum(sp.charge * workloads.E_CHARGE * n[k] for k, sp in enumerate(p.species))
            b = torch.where(self.fixed, self.phi_d * gain, rho * self.volume / workloads.EPS0 + self.lift * gain)
            phi = self.solve(self.systems[0], b, torch.where(self.fixed, self.phi_d * gain, phi))
            phis.append(phi)
            field = -self.gradient(phi)
            size = field.norm(dim=-1)
            mu = []
            for sp in p.species:
                q = sp.mob_params
                mu.append(torch.full_like(size, q[0]) if sp.mob_model == workloads.MOB_CONST
                          else q[0] * (size.clamp(min=q[3]) / q[1]) ** q[2])
            vel = [math.copysign(1.0, sp.charge) * mu[k][:, None] * field for k, sp in enumerate(p.species)]
            src = self.sources(n, size, mu, guesses)
            dt = self.time_step(n, mu, vel, src[p.source.idx[0]])
            new = []
            for k, sp in enumerate(p.species):
                grad = self.gradient(n[k])
                f = self.flux(n[k], grad, vel[k], sp.D, dt)
                gone = n[k][:, None] * vel[k] - (sp.D * grad if sp.bnd_mode == workloads.BND_OUTFLOW else 0.0)
                change = self.scatter(self.hi, f) - self.scatter(self.lo, f) - (gone * self.rim).sum(-1)
                new.append(n[k] + dt * (change / self.volume + src[k]))
            n, t = new, t + dt
        return n, phis, t
