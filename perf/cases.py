"""The calls that users of the IUGKP solver make, as measurable cases: the transport sweep on
1D, 2D and 3D grids (FP64 and FP32 tracking, FP64 and compensated FP32 tallies, gray and
band-resolved), the macro update with the Newton correction, the persistent population, and
whole calls (steady solve, adjoint gradient, statistical averaging).

exact() follows the same particles in 64 bits with torch alone: its own Philox, the straight
flights cell by cell in closed form, and a conjugate-gradient solve of the diffusion equation."""
import math

import numpy as np
import torch

from paper_2506_09465_gb300 import workloads as WL

CHUNK = 1 << 21  # particles followed at a time by exact()


def listed():
    return [
        # A thin film as in the first validation runs: the smallest call, all latency.
        {"name": "sweep_slab_fp64", "kind": "sweep", "geometry": "slab", "n": 50, "kn": 1.0, "particles": 1000,
         "precision": 0, "tally": 0},
        # The rectangle with a heated wall segment at its published particle count: a small
        # fast-path sweep, where launches and the passes around the trace count.
        {"name": "sweep_rectangle", "kind": "sweep", "geometry": "rectangle", "n": 100, "ny": 50, "kn": 10.0,
         "particles": 200, "precision": 1, "tally": 1},
        # The benchmark's square cavity at four Knudsen numbers in one batch: the ordinary sweep.
        {"name": "sweep_cavity4", "kind": "sweep", "geometry": "cavity", "n": 128, "inst": 4, "kn": 0.01,
         "particles": 1024, "precision": 1, "tally": 1},
        # Band-resolved silicon-like square, 80 band-branches, faces beyond the shared window.
        {"name": "sweep_nongray", "kind": "sweep", "geometry": "nongray", "n": 256, "bands": 40, "particles": 1024,
         "precision": 1, "tally": 1},
        # Two-material boxes of uneven sizes up to 64^3: long chains of null candidates.
        {"name": "sweep_boxes", "kind": "sweep", "geometry": "boxes", "inst": 4, "n": 64, "particles": 256,
         "precision": 1, "tally": 1},
        # The FP64 path in earnest: the reference solution that the fast path is compared with.
        {"name": "sweep_cavity_fp64", "kind": "sweep", "geometry": "cavity", "n": 128, "inst": 1, "kn": 1.0,
         "particles": 1024, "precision": 0, "tally": 0},
        # Macro update + Newton correction that close an iteration: separable operator, four squares.
        {"name": "close_cavity4", "kind": "close", "geometry": "cavity", "n": 128, "inst": 4, "kn": 0.01,
         "particles": 1024},
        # The same where the conductivity varies: multigrid-preconditioned CG on the boxes.
        {"name": "close_boxes", "kind": "close", "geometry": "boxes", "inst": 4, "n": 64, "particles": 256},
        # The paper's own persistent population: a reset and its first iterations.
        {"name": "persistent_cavity", "kind": "persistent", "geometry": "cavity", "n": 128, "inst": 1, "kn": 1.0,
         "particles": 1024, "precision": 1, "steps": 8},
        # Adjoint gradient of a hotspot temperature on band-resolved squares of uneven sizes.
        {"name": "adjoint_nongray", "kind": "adjoint", "geometry": "nongray_batch", "inst": 6, "n": 192, "bands": 20,
         "particles": 128},
        # Time to steady state of the benchmark's batch: the whole frozen-draw Newton solve.
        {"name": "solve_cavity4", "kind": "solve", "geometry": "cavity", "n": 128, "inst": 4, "kn": 0.01,
         "particles": 1024, "tol": 1e-8},
        # Averaging after convergence with fresh draws: many small iterations in a row.
        {"name": "average_rectangle", "kind": "average", "geometry": "rectangle", "n": 100, "ny": 50, "kn": 10.0,
         "particles": 200, "steps": 20},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["sweep", "sweep", "sweep", "close", "persistent", "adjoint", "solve", "average"])
    geometry = rng.choice({"sweep": ["slab", "film", "rectangle", "cavity", "nongray", "boxes"],
                           "close": ["film", "cavity", "boxes", "nongray_batch"],
                           "persistent": ["film", "cavity"],
                           "adjoint": ["cavity", "nongray_batch"],
                           "solve": ["slab", "cavity", "nongray"],
                           "average": ["slab", "rectangle"]}[kind])
    c = {"kind": kind, "geometry": geometry}
    if geometry in ("slab", "film"):
        c["n"] = int(_log(rng, 20, 400))
        c["particles"] = int(_log(rng, 200, 8000))
        if geometry == "slab":
            c["kn"] = round(_log(rng, 0.1, 10.0), 3)
    elif geometry == "rectangle":
        c["n"], c["ny"] = int(_log(rng, 15, 160)), int(_log(rng, 15, 120))
        c["kn"] = round(_log(rng, 0.1, 10.0), 3)
        c["particles"] = int(_log(rng, 100, 1500))
    elif geometry == "cavity":
        c["n"] = int(_log(rng, 24, 260 if kind == "close" else 150))
        c["inst"] = rng.choice([1, 1, 2, 3])
        c["kn"] = round(_log(rng, 0.03, 10.0 if c["inst"] == 1 else 0.1), 3)  # ten times more in each next instance
        c["particles"] = int(_log(rng, 64, 1024))
    elif geometry == "nongray":
        c["n"] = int(_log(rng, 40, 256))
        c["bands"] = rng.randint(4, 40)
        c["particles"] = int(_log(rng, 2 * c["bands"] + 16, 1024))
    elif geometry == "nongray_batch":
        c["inst"], c["n"] = rng.randint(2, 6), int(_log(rng, 80, 192))
        c["bands"] = rng.randint(4, 20)
        c["particles"] = 2 * c["bands"] + int(_log(rng, 16, 100))
    else:
        c["inst"], c["n"] = rng.randint(1, 4), int(_log(rng, 16, 48))
        c["particles"] = int(_log(rng, 48, 256))
    if kind == "sweep":
        c["precision"] = 0 if c["geometry"] in ("slab", "rectangle", "cavity") and rng.random() < 0.3 else 1
        c["tally"] = 0 if c["precision"] == 0 else rng.choice([1, 1, 1, 2])
        if c["precision"] == 0:
            c["particles"] = min(c["particles"], 400)
    elif kind == "persistent":
        c["precision"] = rng.choice([0, 1, 1])
        c["steps"] = rng.randint(2, 8)
        if c["precision"] == 0:
            c["particles"] = min(c["particles"], 400)
    elif kind == "solve":
        c["tol"] = 1e-8
        c["particles"] = max(c["particles"], 400)
    elif kind == "average":
        c["steps"] = rng.randint(3, 20)
    return c


# ---- inputs ----------------------------------------------------------------------------------


def _workload(case):
    g, n, N = case["geometry"], case["n"], case["particles"]
    if g == "slab":
        return WL.slab(n, case["kn"], particles=N)
    if g == "film":
        return WL.multiscale_slab(n, particles=N)
    if g == "rectangle":
        return WL.hot_segment_rectangle(case["kn"], n, case["ny"], N)
    if g == "cavity":
        return WL.cavity_sweep(n, [case["kn"] * 10.0 ** i for i in range(case["inst"])], N)
    if g == "nongray":
        return WL.nongray_square(n, case["bands"], N)
    if g == "nongray_batch":
        return WL.nongray_batch(case["inst"], 64, n, case["bands"], N)
    sizes = [int(round(16 + (n - 16) * i / max(1, case["inst"] - 1))) for i in range(case["inst"])]
    return WL.Workload("boxes", np.array([1.0]), np.array([1.0]), [WL.two_material_box(k) for k in sizes], N, N)


def _fields(wl, seed):
    """Cell temperatures of all instances: smooth, within the walls' range, with cell noise."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    out = []
    for inst in wl.instances:
        n = list(inst.n)[: inst.dim]
        axes = [(torch.arange(m, device="cuda", dtype=torch.float64) + 0.5) / m for m in reversed(n)]
        grid = torch.meshgrid(*axes, indexing="ij")
        p = torch.rand(4, generator=gen, device="cuda", dtype=torch.float64)
        T = 0.35 + 0.15 * torch.sin(3.0 * grid[-1] + 6.28 * p[0]) + 0.1 * torch.cos(4.0 * grid[0] + 6.28 * p[1])
        T = T + 0.04 * (torch.rand(T.shape, generator=gen, device="cuda", dtype=torch.float64) - 0.5)
        out.append(T.reshape(-1))
    return torch.cat(out)


def _absorbed(wl, T, seed):
    """Real-collision power [instance][band][cell] as a sweep returns it: the emitted power of a
    field a little off T, with the noise of the particle count."""
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    out, off = [], 0
    for inst in wl.instances:
        nc = inst.ncells
        V = float(np.prod([inst.L[a] / inst.n[a] for a in range(inst.dim)]))
        m = torch.as_tensor(wl.C[:, None] / inst.tau, device="cuda") * V
        x = torch.arange(nc, device="cuda", dtype=torch.float64) / nc
        near = T[off:off + nc] * (1.0 + 0.1 * torch.sin(3.1416 * x))
        noise = torch.randn(m.shape, generator=gen, device="cuda", dtype=torch.float64)
        out.append((m * near[None] * (1.0 + noise / math.sqrt(wl.particles_per_cell))).reshape(-1))
        off += nc
    return torch.cat(out)


def _options(case, seed):
    o = {"seed": seed}
    if case["kind"] in ("sweep", "persistent"):
        o["precision"] = case["precision"]
        if case["precision"] == 0:
            o.update(tally=0, schedule=0)
        elif case["kind"] == "sweep":
            o["tally"] = case["tally"]
    elif case["kind"] == "average":
        o["newton"] = 0
    return o


def _objective(wl):
    return torch.as_tensor(np.concatenate([WL.hotspot_objective(i) for i in wl.instances]), device="cuda")


def prepare(case, seed):
    from paper_2506_09465_gb300.solver import GridSpec, Solver
    wl = _workload(case)
    N = wl.particles_per_cell
    s = Solver([GridSpec(i.dim, i.n, i.L) for i in wl.instances], [i.tau for i in wl.instances], wl.C, wl.v,
               [i.wall_T for i in wl.instances], [i.source for i in wl.instances], particles_per_cell=N,
               particles_per_wall_face=N, **_options(case, seed))
    if any(i.wall_face_T is not None for i in wl.instances):
        s.set_wall_face_T(np.concatenate([i.face_temperatures() for i in wl.instances]))
    st = {"case": case, "solver": s, "T": _fields(wl, seed)}
    if case["kind"] == "close":
        st["R"] = _absorbed(wl, st["T"], seed)
    elif case["kind"] == "adjoint":
        st["g"] = _objective(wl)
    return st


def run(st):
    case, s = st["case"], st["solver"]
    kind = case["kind"]
    if kind == "sweep":
        return s.sweep(st["T"], 3)
    if kind == "close":
        T_half, _ = s.macro(st["R"])
        iters = s.newton_step(st["T"], T_half, st["R"])
        return {"T": T_half, "iters": iters}
    if kind == "persistent":
        s.persistent_reset()
        out = {}
        for it in range(case["steps"]):
            out = s.persistent_step(st["T"], it)
        return out
    if kind == "adjoint":
        grad_source, grad_wall, lam = s.adjoint(st["g"], 1e-8)
        return {"grad_source": grad_source, "grad_wall": grad_wall, "lambda": lam}
    if kind == "solve":
        T, iters, _ = s.solve_steady(st["T"], case["tol"])
        return {"T": T, "iters": iters}
    T = st["T"].clone()
    mean, var, flux = s.average(T, case["steps"], 5, True, True)
    return {"last": T, "mean": mean, "var": var, "flux": flux}


def work(case):
    """Arrays read and written once, and the events of the particles (per flight 200 operations,
    per candidate 50, per face crossed 10, as in a cell-by-cell walk), from the mean free paths."""
    wl = _workload(case)
    nb, by, fl, cells = len(wl.C), 0.0, 0.0, 0
    for inst in wl.instances:
        nc, n = inst.ncells, max(inst.n[: inst.dim])
        h = min(inst.L[a] / inst.n[a] for a in range(inst.dim))
        cells += nc
        faces = sum(nc // inst.n[a] * (inst.n[a] + 1) for a in range(inst.dim))
        by += 8 * (nc + 3 * nb * nc + faces)
        share = wl.C / inst.tau.mean(1)
        share = share / share.sum()
        path = np.minimum(wl.v * inst.tau.mean(1) / h, 0.6 * n)
        cand = np.minimum(inst.tau.mean(1) / inst.tau.min(1), n)
        fl += wl.particles_per_cell * nc * float((share * (200 + 50 * cand + 10 * inst.dim * path)).sum())
    k = case["kind"]
    if k == "close":
        return {"bytes": 8.0 * (nb + 4 + len(wl.instances[0].n)) * cells, "flops": 200.0 * cells}
    if k == "persistent":
        slots = wl.particles_per_cell * cells
        return {"bytes": case["steps"] * (8.0 * slots + by), "flops": case["steps"] * 200.0 * slots}
    times = {"sweep": 1, "adjoint": 8, "solve": 8}.get(k) or case["steps"]
    return {"bytes": times * by, "flops": times * fl}


# ---- the same in 64 bits ---------------------------------------------------------------------

M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, k0, k1):
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57  # low 64 bits; the high word by a masked shift
        c0, c1, c2, c3 = (((p1 >> 32) & M32) ^ c1 ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c3 ^ k1, p0 & M32)
    return c0, c1, c2, c3


def _u(w):
    return ((w >> 9) * 2 + 1).double() * 2.0 ** -24


def _split(N, r):
    r = np.asarray(r, dtype=np.float64)
    share = (N - len(r)) * r / r.sum()
    whole = np.floor(share).astype(np.int64)
    out = 1 + whole
    for j in np.argsort(-(share - whole), kind="stable")[: N - len(r) - int(whole.sum())]:
        out[j] += 1
    return out


class _Instance:
    """One instance's coefficients, and its particles followed in 64 bits."""

    def __init__(self, wl, inst, k, seed):
        self.inst, self.dim, self.k, self.seed = inst, inst.dim, k, seed
        self.n = list(inst.n[: inst.dim]) + [1] * (3 - inst.dim)
        self.L = [inst.L[a] / inst.n[a] if a < inst.dim else 1.0 for a in range(3)]
        self.V = self.L[0] * self.L[1] * self.L[2]
        self.nc = inst.ncells
        self.C, self.v, self.nb = wl.C, wl.v, len(wl.C)
        N = wl.particles_per_cell
        self.n_band = _split(N, wl.C * (1.0 / inst.tau).mean(1))
        self.n_wall = _split(N, wl.C * wl.v)
        self.tau = torch.as_tensor(inst.tau, device="cuda")
        self.C_d = torch.as_tensor(wl.C, device="cuda")
        self.m = (self.C_d[:, None] / self.tau).sum(0)
        src = inst.source if inst.source is not None else np.zeros(self.nc)
        self.shift = torch.as_tensor(src, device="cuda") / self.m
        self.tmaj = inst.tau.min(1)
        self.wall_T = torch.as_tensor(inst.face_temperatures(), device="cuda")
        n = self.n
        self.fax = [0, (n[0] + 1) * n[1] * n[2]]
        self.fax.append(self.fax[1] + (n[0] * (n[1] + 1) * n[2] if self.dim > 1 else 0))
        self.nfaces = self.fax[2] + (n[0] * n[1] * (n[2] + 1) if self.dim > 2 else 0)

    def face(self, a, c):
        """Index of the face normal to a at coordinates c (c[a]: the face's)."""
        m = [self.n[b] + (b == a) for b in range(3)]
        return self.fax[a] + c[0] + m[0] * (c[1] + m[1] * c[2])

    def groups(self, walls=True):
        """Runs of particles: (band, wall or -1, emitters, particles of each, first wall face)."""
        for b in range(self.nb):
            yield b, -1, self.nc, int(self.n_band[b]), 0
        for b in range(self.nb if walls else 0):
            off = 0
            for w in range(2 * self.dim):
                nf = self.n[(w // 2 + 1) % 3] * self.n[(w // 2 + 2) % 3]
                yield b, w, nf, int(self.n_wall[b]), off
                off += nf

    def emit(self, b, w, e, q, epoch):
        n = self.n
        key = (self.seed & M32, ((self.seed >> 32) & M32) ^ self.k)
        top = (b << 24) | (epoch & 0xFFFFFF)
        if w < 0:
            idx = [e % n[0], (e // n[0]) % n[1], e // (n[0] * n[1])]
            ident, face = e, None
        else:
            a = w // 2
            idx = [None] * 3
            idx[a] = torch.full_like(e, n[a] - 1 if w % 2 else 0)
            idx[(a + 1) % 3], idx[(a + 2) % 3] = e % n[(a + 1) % 3], e // n[(a + 1) % 3]
            f = list(idx)
            f[a] = idx[a] + w % 2
            face = self.face(a, f)
            ident = self.nc + face

        def block(k, rows=slice(None)):
            return _philox(torch.zeros_like(ident[rows]) + k, q[rows], ident[rows], torch.full_like(ident[rows], top), *key)

        z = block(0)
        first = (((z[0] & 511) << 14) | ((z[1] & 511) << 5) | ((z[2] & 511) >> 4)) << 9
        xi, s = [None] * 3, [None] * 3
        if w < 0:
            for a in range(self.dim):
                xi[a] = _u(z[a])
            mu = 2.0 * _u(z[self.dim] if self.dim < 3 else z[3]) - 1.0
            phi = _u(z[3]) if self.dim == 2 else (_u(block(1)[0]) if self.dim == 3 else None)
            s[0] = mu
            if self.dim > 1:
                sn, ang = torch.sqrt(1.0 - mu * mu), 2.0 * math.pi * phi
                s[1], s[2] = sn * torch.cos(ang), sn * torch.sin(ang)
            j0 = (2, 4, 6)[self.dim - 1]
        else:
            tang = [a2 for a2 in range(self.dim) if a2 != w // 2]
            for i, a2 in enumerate(tang):
                xi[a2] = _u(z[i])
            un = _u(z[len(tang)])
            xi[w // 2] = torch.full_like(un, float(w % 2))
            s[w // 2] = torch.sqrt(un) * (-1.0 if w % 2 else 1.0)
            if self.dim > 1:
                sn, ang = torch.sqrt(1.0 - un), 2.0 * math.pi * _u(z[len(tang) + 1])
                s[(w // 2 + 1) % 3], s[(w // 2 + 2) % 3] = sn * torch.cos(ang), sn * torch.sin(ang)
            j0 = 2 if self.dim == 1 else 4
        return idx, xi, s, face, first, j0, block

    def follow(self, b, w, e, q, epoch, weight=None, out=None):
        """Cell of the real collision of each particle, -1 at a wall. With weight: its tallies
        into out (R, W of the band, F, wall)."""
        dim, n = self.dim, self.n
        idx, xi, s, face, first, j0, block = self.emit(b, w, e, q, epoch)
        t, d, m, step, tex, ex = [], [], [], [], None, None
        for a in range(dim):
            st = torch.where(s[a] > 0, 1, -1)
            da = self.L[a] / s[a].abs()
            ta = torch.where(s[a] > 0, 1.0 - xi[a], xi[a]) * self.L[a] / s[a].abs()
            ma = torch.where(s[a] > 0, n[a] - idx[a], idx[a] + 1)
            tw = ta + (ma - 1) * da
            ex = torch.zeros_like(idx[a]) if a == 0 else torch.where(tw < tex, a, ex)
            tex = tw if a == 0 else torch.minimum(tex, tw)
            t.append(ta), d.append(da), m.append(ma), step.append(st)
        ratio = float(self.tmaj[b]) / self.tau[b]
        real = bool((ratio == 1.0).all())
        D = -torch.log(_u(first)) * float(self.v[b]) * float(self.tmaj[b])
        cell = torch.full_like(e, -1)
        rows = torch.arange(len(e), device="cuda")  # particles still flying
        k, words = 0, None
        while len(rows):
            rows = rows[D[rows] <= tex[rows]]
            at = torch.zeros_like(rows)
            mul = 1
            for a in range(dim):
                c = torch.ceil((D[rows] - t[a][rows]) / d[a][rows]).clamp(min=0).long()
                at += mul * (idx[a][rows] + step[a][rows] * torch.minimum(c, m[a][rows] - 1))
                mul *= n[a]
            if out is not None:
                out["W"][b].index_add_(0, at, weight[rows] * float(self.tmaj[b]))
            if real:
                cell[rows] = at
                break
            J = j0 + (2 * k + 1 if k else 0)
            ok = _u(block(J // 4, rows)[J % 4]) < ratio[at]
            cell[rows[ok]] = at[ok]
            rows, k = rows[~ok], k + 1
            words = block((j0 + 2 * k) // 4, rows)
            D[rows] += -torch.log(_u(words[(j0 + 2 * k) % 4])) * float(self.v[b]) * float(self.tmaj[b])
        if out is None:
            return cell
        hit = cell >= 0
        out["R"][b].index_add_(0, cell[hit], weight[hit])
        end = torch.where(hit, D, tex)
        if face is not None:
            out["F"].index_add_(0, face, weight * (-1.0 if w % 2 else 1.0))
        for a in range(dim):
            # faces normal to a before the end, the wall's too where the particle leaves there
            c = torch.minimum(torch.ceil((end - t[a]) / d[a]).clamp(min=0).long(), m[a] - 1)
            gone = ~hit & (ex == a)
            c = torch.where(gone, m[a], c)
            out["wall"].index_add_(0, 2 * a + (step[a][gone] > 0).long(), weight[gone])
            p = torch.repeat_interleave(torch.arange(len(c), device="cuda"), c)
            i = torch.arange(len(p), device="cuda") - (torch.cumsum(c, 0) - c)[p]
            T = t[a][p] + i * d[a][p]
            co = [torch.zeros_like(p)] * 3
            for o in range(dim):
                if o == a:
                    co[o] = torch.where(step[a][p] > 0, idx[a][p] + 1 + i, idx[a][p] - i)
                else:
                    x = torch.ceil((T - t[o][p]) / d[o][p]).clamp(min=0).long()
                    co[o] = idx[o][p] + step[o][p] * torch.minimum(x, m[o][p] - 1)
            out["F"].index_add_(0, self.face(a, co), weight[p] * step[a][p])
        return cell

    def particles(self, epoch, walls=True):
        for b, w, ne, per, off in self.groups(walls):
            for p0 in range(0, ne * per, CHUNK):
                p = torch.arange(p0, min(ne * per, p0 + CHUNK), device="cuda")
                yield b, w, p % ne, p // ne, off

    def coefficient(self, b, w, e):
        """Power of a particle per unit temperature of its emitter."""
        if w < 0:
            return self.C[b] * self.V / (self.tau[b][e] * float(self.n_band[b]))
        area = self.V / self.L[w // 2]
        return torch.full_like(e, 1, dtype=torch.float64) * (self.C[b] * self.v[b] * area / (4.0 * float(self.n_wall[b])))

    def sweep(self, T, epoch):
        z = dict(dtype=torch.float64, device="cuda")
        out = {"R": torch.zeros(self.nb, self.nc, **z), "W": torch.zeros(self.nb, self.nc, **z),
               "F": torch.zeros(self.nfaces, **z), "wall": torch.zeros(2 * self.dim, **z)}
        Te = T + self.shift
        for b, w, e, q, off in self.particles(epoch):
            power = Te[e] if w < 0 else self.wall_T[off + e]
            if w >= 0 and not bool((power != 0).any()):
                continue
            self.follow(b, w, e, q, epoch, self.coefficient(b, w, e) * power, out)
        return out

    def map(self, epoch):
        """The sweep as a linear map: emitter (cells, then wall faces), collision cell and power
        per unit emission temperature of every particle that collides."""
        src, dst, co = [], [], []
        for b, w, e, q, off in self.particles(epoch):
            cell = self.follow(b, w, e, q, epoch)
            hit = cell >= 0
            src.append((e if w < 0 else self.nc + off + e)[hit].int())
            dst.append(cell[hit].int())
            co.append(self.coefficient(b, w, e)[hit])
        return torch.cat(src), torch.cat(dst), torch.cat(co)

    def diffusion(self):
        """-div(kappa grad) with the vacuum wall condition, as a function; its diagonal; the
        correction's damping."""
        kap = (self.C_d[:, None] * torch.as_tensor(self.v, device="cuda")[:, None] ** 2 * self.tau / 3.0).sum(0)
        kap = kap.reshape(self.n[2], self.n[1], self.n[0])
        cv, parts, diag = float((self.C * self.v).sum()), [], torch.zeros_like(kap)
        for a in range(self.dim):
            ax, h = 2 - a, self.L[a]
            lo, hi = kap.narrow(ax, 0, self.n[a] - 1), kap.narrow(ax, 1, self.n[a] - 1)
            g = 2.0 * lo * hi / (lo + hi) / h ** 2
            diag.narrow(ax, 0, self.n[a] - 1).add_(g)
            diag.narrow(ax, 1, self.n[a] - 1).add_(g)
            for end in (0, self.n[a] - 1):
                k = kap.narrow(ax, end, 1)
                diag.narrow(ax, end, 1).add_(1.0 / (h / (2.0 * k) + 2.0 / cv) / h)
            parts.append((ax, self.n[a] - 1, g))

        def apply(x):
            x = x.reshape(kap.shape)
            y = diag * x
            for ax, cnt, g in parts:
                y.narrow(ax, 0, cnt).sub_(g * x.narrow(ax, 1, cnt))
                y.narrow(ax, 1, cnt).sub_(g * x.narrow(ax, 0, cnt))
            return y.reshape(-1)

        thick = float((min(self.L[: self.dim]) / torch.sqrt(3.0 * kap.reshape(-1) / self.m)).max())
        return apply, diag.reshape(-1), min(1.0, 1.5 / thick)

    def correction(self, rhs, rtol):
        apply, diag, _ = self.op
        x, r = torch.zeros_like(rhs), rhs.clone()
        z = r / diag
        p, rz, stop = z.clone(), (r * z).sum(), rtol * rhs.norm()
        for it in range(20000):
            q = apply(p)
            al = rz / (p * q).sum()
            x += al * p
            r -= al * q
            if it % 16 == 15 and r.norm() <= stop:
                break
            z = r / diag
            new = (r * z).sum()
            p, rz = z + (new / rz) * p, new
        return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "persistent":
        return None  # single-precision positions carried through the iterations: 64 bits follow other particles
    wl = _workload(case)
    ins = [_Instance(wl, inst, k, seed) for k, inst in enumerate(wl.instances)]
    off = np.cumsum([0] + [i.nc for i in ins])
    T = _fields(wl, seed)
    if kind == "sweep":
        got = [i.sweep(T[off[k]:off[k + 1]], 3) for k, i in enumerate(ins)]
        out = {key: torch.cat([g[key].reshape(-1) for g in got]) for key in ("R", "W", "F", "wall")}
        return {**out, "counters": None}
    if kind == "close":
        R, b0, out = _absorbed(wl, T, seed), 0, []
        for k, i in enumerate(ins):
            i.op = i.diffusion()
            r = R[b0:b0 + i.nb * i.nc].reshape(i.nb, i.nc).sum(0)
            b0 += i.nb * i.nc
            dT = i.correction((r - T[off[k]:off[k + 1]] * i.V * i.m) / i.V, 1e-13)
            out.append(r / (i.V * i.m) + i.op[2] * dT)
        return {"T": torch.cat(out), "iters": None}
    if kind == "average":
        i, mean, m2, flux = ins[0], 0.0, 0.0, 0.0
        for k in range(case["steps"]):
            g = i.sweep(T, 5 + k)
            T = g["R"].sum(0) / (i.V * i.m)
            dev = T - mean
            mean = mean + dev / (k + 1)
            m2, flux = m2 + dev * (T - mean), flux + g["F"]
        return {"last": T, "mean": mean, "var": m2 / (case["steps"] - 1), "flux": flux / case["steps"]}
    outs, g = [], _objective(wl) if kind == "adjoint" else None
    for k, i in enumerate(ins):
        i.op = i.diffusion()
        src, dst, co = i.map(0)
        th, Vm, ne = i.op[2], i.V * i.m, i.nc + len(i.wall_T)
        x = T[off[k]:off[k + 1]] if kind == "solve" else torch.zeros(i.nc, dtype=torch.float64, device="cuda")
        back = lambda lam: torch.zeros(ne, dtype=torch.float64, device="cuda").index_add_(0, src, co * (lam / Vm)[dst])  # noqa: E731
        for _ in range(400):
            if kind == "solve":
                emit = torch.cat([x + i.shift, i.wall_T])
                r = torch.zeros_like(x).index_add_(0, dst, co * emit[src])
                new = r / Vm + th * i.correction((r - x * Vm) / i.V, 1e-4)
            else:
                half = back(x)[: i.nc] + g[off[k]:off[k + 1]]
                new = half + th * i.m * i.correction(half - x, 1e-4)
            far = float((new - x).norm() / new.norm())
            x = new
            if far < 1e-13:
                break
        if kind == "solve":
            outs.append({"T": x})
        else:
            at = back(x)
            nf = [i.n[(w // 2 + 1) % 3] * i.n[(w // 2 + 2) % 3] for w in range(2 * i.dim)]
            outs.append({"grad_source": at[: i.nc] / i.m, "grad_wall": torch.stack([p.sum() for p in at[i.nc:].split(nf)]),
                         "lambda": x})
    out = {key: torch.cat([o[key] for o in outs]) for key in outs[0]}
    return {**out, "iters": None} if kind == "solve" else out
