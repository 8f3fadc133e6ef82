"""Measured cases: what a user of the library has it do, from the smallest
plate to a batch of many, each through the public entry points.

A pass is one solve on a handle the program keeps: back to rest, all time
steps, and the fields (displacement, velocity, stress) on the device.  The
handle is what a program that solves several load cases on one part keeps; the
loads come from the seed.  Sizes and step counts are those of the benchmark
configurations and parity tests, or odd sizes beside them; step counts stay
where the scheme is stable in exact arithmetic.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2208_04088_gb300 import _native as N
from paper_2208_04088_gb300 import workloads as W

NONPOISSON = W.CRACK_PAPER_LAM_OVER_MU

# floating operations of one lattice update: moments 24, relaxation 26,
# populations 30, displacement 11 (FMA = 2)
FLOPS_PER_UPDATE = 91


def _solve(name, kind, nx, ny, steps, **kw):
    c = dict(name=name, form="solve", kind=kind, nx=nx, ny=ny, steps=steps, radius=0.0, length=0,
             lam=1.0, storage="f32", wall_node=True, in_place=False)
    c.update(kw)
    return c


def listed():
    return [
        # the method check: a clamped plate under a suddenly applied traction, the
        # paper's extrapolated wall values; bound by launches, not by bytes
        _solve("square_64", "square", 64, 64, 500, wall_node=False),
        # the small plate with a hole of the parity tests
        _solve("hole_256x128", "hole", 256, 128, 500, radius=16.0),
        # odd sizes and every kind of boundary condition on one plate: moving
        # wall, rigid inclusion, stress, ramped pressure and traction
        _solve("ragged_333x217", "rules", 333, 217, 300, radius=23.5),
        # the paper's own crack run: centre crack, its material (lambda != mu)
        _solve("centre_crack_400", "centre_crack", 400, 400, 210, length=100, lam=NONPOISSON,
               wall_node=False),
        # the plate with a hole at its benchmark size, resident in L2
        _solve("hole_1024x512", "hole", 1024, 512, 600, radius=64.0),
        # the headline: an edge crack in a lattice larger than L2
        _solve("crack_2048", "edge_crack", 2048, 2048, 500, length=512),
        # a large plate with a curved wall under the paper's extrapolation
        _solve("hole_2048_extrapolated", "hole", 2048, 2048, 300, radius=256.0, wall_node=False),
        # the same crack in the 16-bit form, in one buffer, and in the paper's material
        _solve("crack_2048_f16", "edge_crack", 2048, 2048, 500, length=512, storage="f16"),
        _solve("crack_2048_in_place", "edge_crack", 2048, 2048, 500, length=512, in_place=True),
        _solve("crack_2048_nonpoisson", "edge_crack", 2048, 2048, 500, length=512, lam=NONPOISSON),
        # a parameter study: many plates with holes of mixed sizes stepped together
        dict(name="batch_40_f32", form="batch", count=40, pick=4, steps=256, storage="f32"),
        dict(name="batch_40_f16", form="batch", count=40, pick=4, steps=256, storage="f16"),
    ]


def draw(rng):
    if rng.random() < 0.15:
        return dict(form="batch", count=rng.randint(3, 24), pick=rng.randint(0, 10 ** 6),
                    steps=rng.randint(100, 256), storage=rng.choice(["f32", "f32", "f16", "bf16"]))
    kind = rng.choice(["square", "hole", "rules", "edge_crack", "centre_crack"])
    nx = int(math.exp(rng.uniform(math.log(48), math.log(2048))))
    ny = max(40, min(2048, int(nx * math.exp(rng.uniform(math.log(0.5), math.log(1.5))))))
    if kind in ("edge_crack", "centre_crack"):
        ny -= ny % 2  # the crack lies between two rows
    small = min(nx, ny)
    radius = math.exp(rng.uniform(math.log(4.0), math.log(small / 5.0)))
    length = rng.randint(max(2, nx // 8), max(3, nx // 3))
    form = rng.choice(["f32", "f32", "f32", "f32", "nonpoisson", "f16", "bf16", "in_place"])
    wall_node = rng.random() < 0.6
    steps = int(math.exp(rng.uniform(math.log(100), math.log(500 if wall_node else 300))))
    steps = max(32, min(steps, int(1e9 / (nx * ny))))
    return _solve_draw(kind, nx, ny, steps, radius, length, form, wall_node)


def _solve_draw(kind, nx, ny, steps, radius, length, form, wall_node):
    c = _solve("", kind, nx, ny, steps, wall_node=wall_node,
               radius=round(radius, 2) if kind in ("hole", "rules") else 0.0,
               length=length if kind in ("edge_crack", "centre_crack") else 0,
               lam=NONPOISSON if form == "nonpoisson" else 1.0,
               storage=form if form in ("f16", "bf16") else "f32", in_place=form == "in_place")
    del c["name"]
    return c


def _batch_sizes(case):
    """(nx, ny, radius) of each plate: sides 128 to 1024, square or 2:1."""
    rng = np.random.default_rng(case["pick"])
    out = []
    for _ in range(case["count"]):
        a = int(rng.choice([128, 256, 512, 1024]))
        ny = a if rng.integers(0, 2) == 0 else a // 2
        out.append((a, ny, float(rng.integers(8, min(a, ny) // 8 + 1))))
    return out


def _workloads(case, seed):
    """The workloads of a case: geometry from the case, loads from the seed."""
    rng = np.random.default_rng(seed)
    if case["form"] == "batch":
        return [W.hole_plate(nx, ny, r, case["steps"], float(rng.uniform(1e-4, 1e-3)))
                for nx, ny, r in _batch_sizes(case)]
    nx, ny, steps, lam = case["nx"], case["ny"], case["steps"], case["lam"]
    load, shear = float(rng.uniform(2e-4, 1e-3)), float(rng.uniform(-3e-4, 3e-4))
    kind = case["kind"]
    if kind == "square":
        w = W.square_plate(nx, steps, load, lam_over_mu=lam)
        w.ny = ny
        w.bcs[1] = W.bc(W.TRACTION, (load, shear))
    elif kind == "hole":
        w = W.hole_plate(nx, ny, case["radius"], steps, load, lam_over_mu=lam)
        w.bcs[0] = W.bc(W.STRESS, (load, 0.3 * shear, shear))
    elif kind == "rules":
        w = W.hole_plate(nx, ny, case["radius"], steps, load, lam_over_mu=lam)
        w.edge_bc = (0, 2, 3, 4)
        w.hole = (w.hole[0], w.hole[1], w.hole[2], 1)
        w.bcs = [W.bc(W.DIRICHLET, (0.2 * load, -0.1 * load)), W.bc(W.DIRICHLET, (0.0, 0.0)),
                 W.bc(W.STRESS, (load, -0.5 * load, shear)),
                 W.bc(W.PRESSURE, (-0.4 * load,), W.RAMP, 60.0),
                 W.bc(W.TRACTION, (0.2 * load, shear), W.RAMP, 25.0)]
    elif kind == "edge_crack":
        w = W.edge_crack(nx, case["length"], steps, load, lam_over_mu=lam, ny=ny)
        w.bcs[0] = W.bc(W.STRESS, (0.2 * shear, 0.1 * load, 0.0))
    else:
        w = W.centre_crack(case["length"], steps, load, lam_over_mu=lam, side=nx)
        w.ny = ny
        w.bcs[0] = W.bc(W.STRESS, (0.2 * shear, 0.1 * load, 0.0))
    w.wall_node = case["wall_node"]
    return [w]


def prepare(case, seed):
    ws = _workloads(case, seed)
    if case["form"] == "batch":
        batch = N.Batch([N.desc_from_workload(w, storage=case["storage"]) for w in ws])
        out = torch.empty(7 * sum(w.nodes for w in ws), dtype=torch.float32, device="cuda")
        return {"batch": batch, "out": out, "nodes": [w.nodes for w in ws], "steps": case["steps"]}
    d = N.desc_from_workload(ws[0], storage=case["storage"], in_place=case["in_place"])
    return {"solver": N.Solver(d), "steps": case["steps"]}


def run(state):
    if "solver" in state:
        s = state["solver"]
        s.reset()
        s.step(state["steps"])
        return s.fields()
    b, lib = state["batch"], N.load()
    b.reset()
    b.step(state["steps"])
    at = state["out"].data_ptr()
    for i, n in enumerate(state["nodes"]):  # every plate's planes u, v, sigma, one after another
        u, v, s = (ctypes.c_void_p(at + 4 * k * n) for k in (0, 2, 4))
        st = lib.lbm_batch_get_fields(b.h, i, u, v, s, 1)
        if st != N.LBM_OK:
            raise N.LbmError(st, N.lbm_last_error())
        at += 28 * n
    return {"fields": state["out"]}


def work(case):
    sizes = (_batch_sizes(case) if case["form"] == "batch"
             else [(case["nx"], case["ny"], case["radius"])])
    box = sum(nx * ny for nx, ny, _ in sizes)
    material = box - sum(math.pi * r * r for _, _, r in sizes)
    # the node mask in, seven field planes out
    return {"bytes": 29.0 * box, "flops": FLOPS_PER_UPDATE * material * case["steps"]}


# ---------------------------------------------------------------------------
# The same solve in 64 bits with plain torch: populations as deviations from
# the rest state, one tensor [9, ny, nx], one step at a time.
_C = np.array([[0, 0], [1, 0], [0, 1], [-1, 0], [0, -1], [1, 1], [-1, 1], [-1, -1], [1, -1]])
_OPP = np.array([0, 3, 4, 1, 2, 7, 8, 5, 6])
_WT = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)


def _mask_and_links(w):
    """Material mask and the columns of the cut links (x, y, direction, wall
    distance q, normal, boundary conditions, corner and curved flags)."""
    nx, ny = w.nx, w.ny
    y, x = np.mgrid[0:ny, 0:nx]
    mat = np.ones((ny, nx), bool)
    if w.hole:
        cx, cy, r, hole_bc = w.hole
        mat = (x - cx) ** 2 + (y - cy) ** 2 >= r * r
    rows = []
    for i in range(1, 9):
        tx, ty = x + _C[i, 0], y + _C[i, 1]
        left, right, below, above = tx < 0, tx >= nx, ty < 0, ty >= ny
        on_crack = np.zeros_like(mat)
        if w.crack and _C[i, 1]:
            x0 = w.crack[2] if len(w.crack) > 2 else 0
            xm = x + 0.5 * _C[i, 0]
            on_crack = ((y + 0.5 * _C[i, 1] == 0.5 * ny - 0.5) & (xm < x0 + w.crack[0] - 0.5) &
                        ((x0 == 0) | (xm > x0 - 0.5)))
        xe, ye = left | right, below | above | on_crack
        end = mat[np.clip(ty, 0, ny - 1), np.clip(tx, 0, nx - 1)]
        for k in np.argwhere(mat & (xe | ye | ~end)):
            k = tuple(k)
            q, n0, n1, bc, bc2, curved = 0.5, 0.0, 0.0, -1, -1, False
            bx = w.edge_bc[0] if left[k] else w.edge_bc[1]
            by = w.crack[1] if on_crack[k] else w.edge_bc[2] if below[k] else w.edge_bc[3]
            if xe[k]:
                n0, bc = float(_C[i, 0]), bx
            if ye[k]:
                n1 = float(_C[i, 1])
                bc, bc2 = (bc, by) if xe[k] else (by, -1)
            if not (xe[k] or ye[k]):
                dx, dy = x[k] - cx, y[k] - cy
                b, a = _C[i, 0] * dx + _C[i, 1] * dy, float((_C[i] ** 2).sum())
                q = (-b - math.sqrt(b * b - a * (dx * dx + dy * dy - r * r))) / a
                n0, n1 = (cx - x[k] - q * _C[i, 0]) / r, (cy - y[k] - q * _C[i, 1]) / r
                bc, curved = hole_bc, True
            rows.append((x[k], y[k], i, q, n0, n1, bc, bc2, curved))
    cols = [np.array(c) for c in zip(*rows)]
    return mat, cols


class _Walls:
    """The boundary rules on all cut links at once."""

    def __init__(self, w, mat, cols):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        x, y, i, q, n0, n1, bc, bc2, curved = cols
        nx, ny = w.nx, w.ny
        cut = np.zeros((9, ny, nx), bool)
        cut[i, y, x] = True
        ux, uy = x - _C[i, 0], y - _C[i, 1]  # the upstream node of the link
        usable = ~cut[_OPP[i], y, x] & (ux >= 0) & (ux < nx) & (uy >= 0) & (uy < ny)
        ux, uy = np.where(usable, ux, x), np.where(usable, uy, y)
        usable &= mat[uy, ux]
        ux, uy = np.where(usable, ux, x), np.where(usable, uy, y)
        kind = np.array([b["kind"] for b in w.bcs] + [-1])
        dirich = (kind[bc] == W.DIRICHLET) | (kind[bc2] == W.DIRICHLET)
        q = np.where(curved & usable, q, 0.5)
        extrapolate = usable & ~dirich & (not w.wall_node)
        t = lambda a, d=torch.float64: torch.as_tensor(np.ascontiguousarray(a), dtype=d, device=dev)
        self.node, self.up = t(y * nx + x, torch.int64), t(uy * nx + ux, torch.int64)
        self.i, self.opp = t(i, torch.int64), t(_OPP[i], torch.int64)
        self.kap, self.fac = t((1 - 2 * q) / (1 + 2 * q)), t(2 / (1 + 2 * q))
        self.kap *= t(usable)
        self.qx = t(np.where(extrapolate, q, 0.0))
        self.wt, self.cx, self.cy = t(_WT[i]), t(_C[i, 0]), t(_C[i, 1])
        self.dirich = t(dirich, torch.bool)
        self.corner = t((bc2 >= 0) & ~dirich, torch.bool)
        self.n0, self.n1 = t(n0), t(n1)
        self.dev = dev
        # boundary data at full amplitude, and the link sets that share a profile
        self.terms = []
        for b, spec in enumerate(w.bcs):
            v = spec["value"]
            for first in (True, False):
                at = (bc if first else bc2) == b
                if not at.any():
                    continue
                cor = bc2 >= 0
                m0 = np.where(cor & (not first), 0.0, n0)  # a corner link's two edges
                m1 = np.where(cor & first, 0.0, n1)
                if spec["kind"] == W.PRESSURE:
                    tx, ty = -v[0] * m0, -v[0] * m1
                elif spec["kind"] == W.STRESS:
                    tx, ty = v[0] * m0 + v[2] * m1, v[2] * m0 + v[1] * m1
                else:
                    tx, ty = v[0] + 0 * m0, v[1] + 0 * m0
                edges = (kind[bc] == W.DIRICHLET).astype(float) + (kind[bc2] == W.DIRICHLET)
                share = np.where(dirich, (spec["kind"] == W.DIRICHLET) / np.maximum(edges, 1.0), 1.0)
                self.terms.append((spec, first, t(at * tx * share), t(at * ty * share)))

    def data(self, time):
        """t* (or d(u*)/dt) of each link's first and second boundary condition."""
        out = [torch.zeros_like(self.kap) for _ in range(4)]
        for spec, first, tx, ty in self.terms:
            amp = min(time / spec["t_ramp"], 1.0) if spec["profile"] == W.RAMP else 1.0
            out[0 if first else 2] += amp * tx
            out[1 if first else 3] += amp * ty
        return out

    def apply(self, w, fcol, mom, fnew, time):
        """fnew at the wall side of every cut link; mom = (drho, Pxx, Pyy, Pxy) planes."""
        g = fcol.reshape(9, -1)
        fi, fo, fu = g[self.i, self.node], g[self.opp, self.node], g[self.i, self.up]
        ax, ay, bx, by = self.data(time)
        cj = w.rho0 * (self.cx * (ax + bx) + self.cy * (ay + by))
        bounce = fi + self.kap * (fu - fo) - self.fac * 6.0 * self.wt * cj
        m = mom.reshape(4, -1)
        at = (1.0 + self.qx) * m[:, self.node] - self.qx * m[:, self.up]
        dr, div = at[0], (w.lam - w.mu) * -at[0] / w.rho0
        sxx, syy, sxy = -at[1] + div, -at[2] + div, -at[3]
        n0, n1 = self.n0, self.n1
        t0, t1 = -n1, n0
        tn, tt = ax * n0 + ay * n1, ax * t0 + ay * t1
        stt = t0 * t0 * sxx + 2 * t0 * t1 * sxy + t1 * t1 * syy
        wxx = tn * n0 * n0 + 2 * tt * n0 * t0 + stt * t0 * t0
        wyy = tn * n1 * n1 + 2 * tt * n1 * t1 + stt * t1 * t1
        wxy = tn * n0 * n1 + tt * (n0 * t1 + t0 * n1) + stt * t0 * t1
        wxx = torch.where(self.corner, ax * n0, wxx)
        wyy = torch.where(self.corner, by * n1, wyy)
        wxy = torch.where(self.corner, 0.5 * (ay * n0 + bx * n1), wxy)
        pxx, pyy, pxy = -wxx + div - dr / 3, -wyy + div - dr / 3, -wxy
        cx, cy = self.cx, self.cy
        second = (cx * cx - 1 / 3) * pxx + (cy * cy - 1 / 3) * pyy + 2 * cx * cy * pxy
        anti = -fi - self.kap * (fu + fo) + self.fac * 2.0 * self.wt * (dr + 4.5 * second)
        fnew.reshape(9, -1)[self.opp, self.node] = torch.where(self.dirich, bounce, anti)


def _collision_matrix(tau):
    """f^col = A f (+ 3 w c.S): BGK towards the equilibrium of f's own moments."""
    c = _C.astype(float)
    eq = np.empty((9, 9))
    for k in range(9):
        p = np.outer(c[k], c[k]) - np.eye(2) / 3
        for i in range(9):
            h = np.outer(c[i], c[i]) - np.eye(2) / 3
            eq[i, k] = _WT[i] * (1 + 3 * c[i] @ c[k] + 4.5 * (p * h).sum())
    return np.eye(9) + (eq - np.eye(9)) / tau


def _solve64(w):
    mat, cols = _mask_and_links(w)
    walls = _Walls(w, mat, cols)
    dev, ny, nx = walls.dev, w.ny, w.nx
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)
    c = _C.astype(float)
    moments = t(np.stack([np.ones(9), c[:, 0] ** 2, c[:, 1] ** 2, c[:, 0] * c[:, 1], c[:, 0], c[:, 1]]))
    both = torch.cat([t(_collision_matrix(w.tau)), moments])
    void = torch.as_tensor(np.flatnonzero(~mat), device=dev)
    grad = w.lam != w.mu
    cut = np.zeros((9, ny, nx), bool)
    cut[cols[2], cols[1], cols[0]] = True
    xp, yp, xm, ym = (t(~cut[d] & mat) for d in (1, 2, 3, 4))  # open axis links
    wcx, wcy = t(3 * _WT * c[:, 0]).view(9, 1, 1), t(3 * _WT * c[:, 1]).view(9, 1, 1)

    def source(dr):
        g = [torch.zeros_like(dr), torch.zeros_like(dr)]
        for a, (p, m, ax) in enumerate(((xp, xm, 1), (yp, ym, 0))):
            up, down = torch.roll(dr, -1, ax) - dr, dr - torch.roll(dr, 1, ax)
            g[a] = (p * up + m * down) / torch.clamp(p + m, min=1.0)
        k = (w.mu - w.lam) / (w.rho0 + dr)
        return k * g[0], k * g[1]

    f = torch.zeros((9, ny, nx), dtype=torch.float64, device=dev)
    u = torch.zeros((2, ny, nx), dtype=torch.float64, device=dev)
    for step in range(w.steps):
        r = (both @ f.view(9, -1)).view(15, ny, nx)
        fcol, mom, jx, jy = r[:9], r[9:13], r[13], r[14]
        if grad:
            sx, sy = source(mom[0])
            fcol += wcx * sx + wcy * sy
            jx, jy = jx + 0.5 * sx, jy + 0.5 * sy
        rho = w.rho0 + mom[0]
        u[0] += jx / rho
        u[1] += jy / rho
        f = torch.empty_like(f)
        for i in range(9):
            f[i] = torch.roll(fcol[i], (int(_C[i, 1]), int(_C[i, 0])), (0, 1))
        walls.apply(w, fcol, mom, f, float(step))
        if len(void):
            f.view(9, -1)[:, void] = 0.0
    mom = (moments @ f.view(9, -1)).view(6, ny, nx)
    jx, jy = mom[4], mom[5]
    if grad:
        sx, sy = source(mom[0])
        jx, jy = jx + 0.5 * sx, jy + 0.5 * sy
    rho, div = w.rho0 + mom[0], (w.lam - w.mu) * -mom[0] / w.rho0
    inside = t(mat)
    return {"u": u * inside, "v": torch.stack([jx / rho, jy / rho]) * inside,
            "sigma": torch.stack([-mom[1] + div, -mom[2] + div, -mom[3]]) * inside}


def exact(case, seed):
    ws = _workloads(case, seed)
    if case["form"] == "batch":
        parts = []
        for w in ws:
            r = _solve64(w)
            parts += [r[k].reshape(-1) for k in ("u", "v", "sigma")]
        return {"fields": torch.cat(parts)}
    return _solve64(ws[0])
