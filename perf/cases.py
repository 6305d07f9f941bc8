"""The calls whose speed counts: what a program that uses this framework spends its time in.

Each case builds a band with its interior boundary (the handle a program keeps), makes inputs from a
seed and runs one public call, or the few calls that belong together.  Sizes are those of the
repository's own workloads: the unit circle at h = 0.01, the unit sphere at h = 1/32 ... 1/256, the
torus R = 1, r = 0.4, the bumpy sphere up to h = 1/640.

`exact` is a plain 64-bit torch restatement of the discrete system (band, interpolation E, crossing
test, difference stencil L, boundary rows), written from the definitions in include/cpm.h.
"""
from __future__ import annotations

import math
import types

import numpy as np
import torch

from paper_2305_04711_gb300.autograd import cpm_solve
from paper_2305_04711_gb300.cpm import Band
from paper_2305_04711_gb300.timestep import heat_cn

DIR1, DIR2 = 1, 2
CIRCLE, SPHERE, TORUS, BUMPY = 1, 2, 3, 4
KIND = {"circle": CIRCLE, "sphere": SPHERE, "torus": TORUS, "bumpy": BUMPY}
TUBE = 0.4  # the torus's minor radius


def _case(name, op, shape, inv_h, p=3, bc=DIR1, dtype="float64", nrhs=1, mode="fp64", steps=1):
    c = {"op": op, "shape": shape, "inv_h": inv_h, "p": p, "bc": bc, "dtype": dtype, "nrhs": nrhs, "mode": mode,
         "steps": steps}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest problem: Laplace-Beltrami on the unit circle between two Dirichlet points, about
        # 5 thousand unknowns; hundreds of iterations whose launches and waits are all there is
        _case("circle_solve", "solve", "circle", 100),
        # time stepping on a coarse sphere: five Crank-Nicolson steps, each a product, a right-hand side
        # and a short warm-started solve
        _case("sphere_heat_steps", "steps", "sphere", 32, steps=5),
        # one backward Euler heat step (dt = h) from a circle of Dirichlet data, the first step of the heat method
        _case("torus_heat_solve", "heat", "torus", 64, bc=DIR2),
        # the matrix-free product of the sphere study in FP64: what a Krylov loop of the caller's own,
        # and every residual of the library's, calls
        _case("sphere_apply_fp64", "apply", "sphere", 128),
        # the largest band (43 million unknowns): the single-precision product that is measured against
        # the memory's bandwidth
        _case("bumpy_apply_fp32", "apply", "bumpy", 640, dtype="float32"),
        # the batched single-precision product, 64 right-hand sides: the inside of the batched refinement solve
        _case("sphere_apply_fp32_x64", "apply", "sphere", 128, dtype="float32", nrhs=64),
        # its double-precision residual, on the torus of the diffusion curves
        _case("torus_apply_fp64_x64", "apply", "torus", 64, nrhs=64),
        # three colour channels of a diffusion-curve image at once
        _case("torus_apply_fp32_x3", "apply", "torus", 128, dtype="float32", nrhs=3),
        # the adjoint's product on the band of the boundary-value fitting workload
        _case("sphere_transpose_fp64", "transpose", "sphere", 256),
        # 64 Poisson problems by FP32 iterations and FP64 refinement, as the batched headline runs them
        _case("sphere_solve_refined_x64", "solve", "sphere", 32, dtype="float64", nrhs=64, mode="fp32_ir"),
        # one step of fitting Dirichlet values to a target: forward solve, loss, adjoint solve, gradients
        _case("sphere_gradient", "gradient", "sphere", 32),
        # the vector-field steps of the heat method on a fine grid: unit gradient, then its divergence
        _case("torus_fields", "fields", "torus", 160),
    ]


# inverse grid spacings an operation is drawn from (per surface: the finest is coarser for the larger ones)
_RANGE = {
    "apply": {"circle": (50, 1000), "sphere": (16, 256), "torus": (20, 200), "bumpy": (24, 400)},
    "transpose": {"circle": (50, 1000), "sphere": (16, 256), "torus": (20, 200)},
    "fields": {"circle": (50, 1000), "sphere": (16, 200), "torus": (20, 160)},
    "solve": {"circle": (50, 200), "sphere": (16, 48), "torus": (20, 32)},
    "heat": {"circle": (50, 200), "sphere": (16, 96), "torus": (20, 64)},
    "steps": {"circle": (50, 200), "sphere": (16, 64), "torus": (20, 48)},
    "gradient": {"sphere": (16, 40), "torus": (20, 28)},
}


def draw(rng):
    """One more call of the same kinds: sizes spread over the logarithm of their ranges, odd ones among
    them, batches from one column to 64, both degrees, both precisions, both orders of the boundary rows."""
    op = rng.choice(["apply", "apply", "apply", "transpose", "fields", "solve", "heat", "steps", "gradient"])
    shape = rng.choice(sorted(_RANGE[op]))
    lo, hi = _RANGE[op][shape]
    inv_h = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    nrhs, dtype, mode = 1, "float64", "fp64"
    if op in ("apply", "transpose"):
        dtype = rng.choice(["float32", "float64"])
        nrhs = rng.choice([1, 1, 1, rng.randint(2, 15), rng.randint(16, 64)])
    elif op == "solve":
        mode = rng.choice(["fp64", "fp32_ir"])
        nrhs = rng.choice([1, 1, rng.randint(2, 15), rng.randint(16, 64)]) if shape != "torus" else 1
        if nrhs > 1 and shape == "sphere":
            inv_h = min(inv_h, 24.0)
    elif op == "heat":
        mode = rng.choice(["fp64", "fp32_ir"])
    if op != "solve" and nrhs > 1 and shape != "circle":  # no dearer than the largest listed batch
        inv_h = min(inv_h, 128.0 if dtype == "float32" else 64.0)
    p, bc = rng.choice([3, 3, 2]), rng.choice([DIR1, DIR2])
    if op == "solve" and shape == "circle":
        # Poisson on the circle at second order is too ill-conditioned for BiCGSTAB at the finer spacings
        p, bc, mode = 3, DIR1, "fp64"
    return _case(None, op, shape, round(inv_h, 2), p=p, bc=bc, dtype=dtype, nrhs=nrhs, mode=mode,
                 steps=rng.randint(2, 6) if op == "steps" else 1)


# ---- what a program has in hand ------------------------------------------------------------------
def _shape(kind):
    s = types.SimpleNamespace(kind=KIND[kind], dim=2 if kind == "circle" else 3, R=1.0, rt=0.0, a=None, c=None, amp=0.1,
                              width=0.05, seed_point=(1.0, 0.0, 0.0))
    if kind == "torus":
        s.rt, s.seed_point = TUBE, (1.0 + TUBE, 0.0, 0.0)
    if kind == "bumpy":  # 16 Gaussian bumps, the repository's bumpy sphere
        r = np.random.default_rng(0)
        s.a = r.uniform(-1.0, 1.0, size=16)
        s.c = r.normal(size=(16, 3))
        s.c /= np.linalg.norm(s.c, axis=1, keepdims=True)
        rho = 1.0 + s.amp * float(np.sum(s.a * np.exp(-np.sum((np.array([1.0, 0.0, 0.0]) - s.c) ** 2, axis=1) / s.width)))
        s.seed_point = (rho, 0.0, 0.0)
    return s


def _curves(kind, bc):
    """Two interior boundaries on each surface (a bumpy sphere takes one point)."""
    def point(p, t):
        return types.SimpleNamespace(kind=1, bc=bc, p=p, nu=t, rad=0.0, ref=(1.0, 0.0, 0.0), two_sided=False)

    def circle(p, nu, rad, ref):
        return types.SimpleNamespace(kind=2, bc=bc, p=p, nu=nu, rad=rad, ref=ref, two_sided=False)

    if kind == "circle":
        return [point((math.cos(a), math.sin(a), 0.0), (-math.sin(a), math.cos(a), 0.0)) for a in (0.1, 0.1 + math.pi / 2)]
    if kind == "sphere":
        return [circle((0.0, 0.0, math.cos(a)), (0.0, 0.0, 1.0), math.sin(a), (1.0, 0.0, 0.0))
                for a in (math.pi / 4, 3 * math.pi / 4)]
    if kind == "torus":
        return [circle((math.cos(a), math.sin(a), 0.0), (-math.sin(a), math.cos(a), 0.0), TUBE,
                       (math.cos(a), math.sin(a), 0.0)) for a in (0.3, 2.5)]
    return []


def _samples(case):
    """Dirichlet samples per curve: one at a point, a ring of them on a circle."""
    return [1, 1] if case["shape"] == "circle" else [64, 64]


def _generator(seed, salt):
    return np.random.default_rng([int(seed), salt])


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _noise(n, nrhs, seed):
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed) * 7919 + 17)
    return torch.randn((n,) if nrhs == 1 else (n, nrhs), generator=g, dtype=torch.float64, device=_device())


def _waves(cp, seed, nrhs, salt=1):
    """Smooth surface fields, as sources, targets and states are: a few plane waves at the closest points."""
    r = _generator(seed, salt)
    out = torch.zeros((cp.shape[0], nrhs), dtype=torch.float64, device=cp.device)
    for _ in range(3):
        k = torch.tensor(r.normal(size=(3, nrhs)) * 1.5, device=cp.device)
        ph = torch.tensor(r.uniform(0, 2 * math.pi, size=nrhs), device=cp.device)
        am = torch.tensor(r.uniform(0.3, 1.0, size=nrhs), device=cp.device)
        out += am * torch.sin(cp @ k + ph)
    return out[:, 0].contiguous() if nrhs == 1 else out


def _inputs(case, seed, cp, twin):
    """The vectors of a case, given the closest points of the PDE unknowns and the twins of the boundary ones."""
    op, nrhs = case["op"], case["nrhs"]
    full = torch.cat([cp, cp[twin]]) if twin.numel() else cp
    tot = sum(_samples(case)) if twin.numel() else 0
    if op in ("apply", "transpose"):  # a Krylov vector: a smooth part and a rough one
        u = _waves(full, seed, nrhs) + 0.25 * _noise(full.shape[0], nrhs, seed)
        return {"u": u.to(getattr(torch, case["dtype"]))}
    if op == "fields":
        return {"u": _waves(full, seed, 1)}
    ring = torch.tensor(_generator(seed, 2).uniform(0.0, 1.0, size=(tot,) if nrhs == 1 else (tot, nrhs)), device=cp.device)
    if op == "solve":  # Poisson with Dirichlet data
        return {"s": _waves(cp, seed, nrhs), "samples": ring}
    if op == "heat":
        return {"samples": ring}
    if op == "steps":
        return {"u": _waves(full, seed, 1), "g": torch.tensor(_generator(seed, 3).uniform(0, 1, size=twin.numel()), device=cp.device)}
    return {"s": _waves(cp, seed, 1), "samples": ring, "target": _waves(full, seed, 1, salt=4)}


def prepare(case, seed):
    h = 1.0 / case["inv_h"]
    curves = _curves(case["shape"], case["bc"])
    band = Band(_shape(case["shape"]), h, p=case["p"])
    band.set_boundary(curves, _samples(case) if curves else None)
    if case["nrhs"] > 1:
        band.reserve(case["nrhs"], fp32_ir=case["mode"] == "fp32_ir" or case["dtype"] == "float32")
    _, cp = band.export_band()
    return {"case": case, "band": band, "h": h, **_inputs(case, seed, cp, band.export_boundary()["twin"])}


def run(state):
    case, band, h = state["case"], state["band"], state["h"]
    op = case["op"]
    if op in ("apply", "transpose"):  # M u, the operator of the Poisson problems
        return band.apply(0.0, 1.0, state["u"], transpose=op == "transpose")
    if op == "fields":
        X = band.surface_gradient(state["u"], normalize=True)
        return X, band.surface_divergence(X)
    if op == "solve":
        f = band.rhs(s=state["s"], samples=state["samples"], nrhs=case["nrhs"])
        return band.solve(0.0, 1.0, f, tol=1e-12, mode=case["mode"])[0]
    if op == "heat":
        return band.solve(1.0, -h, band.rhs(samples=state["samples"]), tol=1e-12, mode=case["mode"])[0]
    if op == "steps":
        return heat_cn(band, state["u"], h, case["steps"], g=state["g"])[0]
    s, samples = state["s"].detach().requires_grad_(), state["samples"].detach().requires_grad_()
    u = cpm_solve(band, 0.0, 1.0, s, samples, tol=1e-11)
    (0.5 * (u - state["target"]).square().sum()).backward()
    return u.detach(), s.grad, samples.grad


# ---- work ---------------------------------------------------------------------------------------
def _rows(case):
    """Unknowns of a band: the tube of radius Eq. (3) around the surface."""
    h, half = 1.0 / case["inv_h"], (case["p"] + 1) / 2.0
    dim = 2 if case["shape"] == "circle" else 3
    r = h * math.sqrt((dim - 1) * half * half + (1 + half) ** 2)
    area = {"circle": 2 * math.pi, "sphere": 4 * math.pi, "torus": 4 * math.pi ** 2 * TUBE, "bumpy": 4.2 * math.pi}[case["shape"]]
    return area * 2 * r / h ** dim


def work(case):
    n, w = _rows(case), 8 if case["dtype"] == "float64" else 4
    m = n * case["nrhs"]
    # a product: input, output, the fractional stencil position and the base of each row; its separable
    # gather and seven-point sum
    dim = 2 if case["shape"] == "circle" else 3
    np1 = case["p"] + 1
    gather = 2 * sum(np1 ** d for d in range(1, dim + 1)) + 12
    product = {"bytes": 2 * w * m + (dim * w + 4) * n, "flops": gather * m + 36 * n}
    if case["op"] in ("apply", "transpose"):
        return product
    if case["op"] == "fields":
        return {"bytes": (8 + 24 + 24 + 8 + 28) * n, "flops": 4 * gather * n}
    # solves: iterations grow like 1/h (Poisson) or its root (a heat step); each has two products and ten
    # vectors that the recurrences read and write.  A refined solve iterates in 32 bits.
    its = {"solve": 8.0, "gradient": 16.0}.get(case["op"], 0) * case["inv_h"] + \
        {"heat": 9.0, "steps": 7.0 * case["steps"]}.get(case["op"], 0) * math.sqrt(case["inv_h"])
    w = 4 if case["mode"] == "fp32_ir" else 8
    return {"bytes": its * (2 * (dim * w + 4) * n + 14 * w * m), "flops": its * (2 * product["flops"] + 20 * m)}


# ---- the same system in plain torch, 64 bits -------------------------------------------------------
def _cp_surface(kind, x):
    if kind == "circle":
        n = torch.sqrt(x[:, 0] * x[:, 0] + x[:, 1] * x[:, 1])
        return torch.stack([x[:, 0] / n, x[:, 1] / n, torch.zeros_like(n)], 1)
    if kind == "sphere":
        return x / torch.sqrt(x[:, 0] * x[:, 0] + x[:, 1] * x[:, 1] + x[:, 2] * x[:, 2])[:, None]
    rho = torch.sqrt(x[:, 0] * x[:, 0] + x[:, 1] * x[:, 1])
    c = torch.stack([x[:, 0] / rho, x[:, 1] / rho, torch.zeros_like(rho)], 1)
    d = x - c
    m = torch.sqrt(d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1] + d[:, 2] * d[:, 2])
    return c + TUBE * (d / m[:, None])


def _dot(a, b):
    return a[..., 0] * b[..., 0] + a[..., 1] * b[..., 1] + a[..., 2] * b[..., 2]


class _System:
    """The discrete system of one case: band, E, L and the boundary rows (include/cpm.h)."""

    def __init__(self, case):
        kind, self.dim, self.p = case["shape"], 2 if case["shape"] == "circle" else 3, case["p"]
        self.h, self.np1 = 1.0 / case["inv_h"], case["p"] + 1
        self.kind, self.bc, self.dev = kind, case["bc"], _device()
        h, half = self.h, (self.p + 1.0) / 2.0
        self.r = h * math.sqrt((self.dim - 1) * (half * half) + (1.0 + half) * (1.0 + half))
        self._band()
        self._curves(case)

    def _band(self):
        h, dev = self.h, self.dev
        ext = (1.0 + (TUBE if self.kind == "torus" else 0.0)) + self.r
        top = TUBE + self.r if self.kind == "torus" else ext
        b, bz = -(-int(ext / h + 2) // 8), -(-int(top / h + 2) // 8) if self.dim == 3 else 0
        self.b, self.bz = b, bz
        ax = torch.arange(-8 * b, 8 * b, device=dev)
        gj, gi = torch.meshgrid(ax, ax, indexing="ij")
        flat = torch.stack([gi.reshape(-1), gj.reshape(-1)], 1)
        found = []
        for k in range(-8 * bz, 8 * bz) if self.dim == 3 else [0]:
            x = torch.zeros((flat.shape[0], 3), dtype=torch.float64, device=dev)
            x[:, :2] = flat.double() * h
            x[:, 2] = k * h
            rough = torch.sqrt(x[:, 0] * x[:, 0] + x[:, 1] * x[:, 1])
            if self.kind == "torus":
                near = (torch.sqrt((rough - 1.0) ** 2 + (k * h) ** 2) - TUBE).abs() < self.r + h
            else:
                near = (torch.sqrt(rough * rough + (k * h) ** 2) - 1.0).abs() < self.r + h
            at = near.nonzero()[:, 0]
            x = x[at]
            cp = _cp_surface(self.kind, x)
            d = x - cp
            keep = torch.sqrt(_dot(d, d)) <= self.r
            at = at[keep]
            found.append((torch.cat([flat[at], torch.full_like(at[:, None], k)], 1), cp[keep]))
        ijk, cp = torch.cat([f[0] for f in found]), torch.cat([f[1] for f in found])
        key = self._key(ijk)
        self.key, order = torch.sort(key)
        self.ijk, self.cp = ijk[order], cp[order]
        self.n = ijk.shape[0]
        self.x = self.ijk.double() * self.h

    def _key(self, g):
        """Canonical order: 8^3 bricks by (z, y, x), then nodes by (z, y, x)."""
        o = torch.tensor([8 * self.b, 8 * self.b, 8 * self.bz], device=g.device)
        q = g + o
        br, lo = q >> 3, q & 7
        return (((br[..., 2] * (2 * self.b) + br[..., 1]) * (2 * self.b) + br[..., 0]) << 9) + lo[..., 2] * 64 + lo[..., 1] * 8 + lo[..., 0]

    def _find(self, g):
        k = self._key(g)
        at = torch.searchsorted(self.key, k).clamp_(max=self.n - 1)
        return torch.where(self.key[at] == k, at, torch.full_like(at, -1))

    def _stencil(self, y):
        """Nodes and weights of the interpolation at points y: [q, np1^dim] each, x fastest."""
        s = y / self.h
        base = (torch.floor(s + 0.5) if self.p == 2 else torch.floor(s)) - 1
        t = s - base
        w = []
        for a in range(self.dim):
            ta = t[:, a]
            w.append(torch.stack([torch.stack([(ta - o) / (q - o) for o in range(self.np1) if o != q]).prod(0)
                                  for q in range(self.np1)], 1))
        base = base.long()
        if self.dim == 2:
            base[:, 2] = 0
        r = range(self.np1)
        off = [(x, y_, z) for z in (r if self.dim == 3 else [0]) for y_ in r for x in r]
        o = torch.tensor(off, device=y.device)
        ww = w[0][:, o[:, 0]] * w[1][:, o[:, 1]]
        if self.dim == 3:
            ww = ww * w[2][:, o[:, 2]]
        return self._find(base[:, None, :] + o), ww

    def _cp_curve(self, cv, x):
        if cv.kind == 1:
            return torch.tensor(cv.p, dtype=torch.float64, device=x.device).expand_as(x)
        p, nu = (torch.tensor(v, dtype=torch.float64, device=x.device) for v in (cv.p, cv.nu))
        w = x - p
        q = w - _dot(w, nu.expand_as(w))[:, None] * nu
        nq = torch.sqrt(_dot(q, q))
        ref = torch.tensor(cv.ref, dtype=torch.float64, device=x.device)
        unit = torch.where((nq == 0)[:, None], ref.expand_as(q), q / nq[:, None])
        return p + cv.rad * unit

    def _curves(self, case):
        dev, n = self.dev, self.n
        self.curves = _curves(self.kind, self.bc)
        self.twin, self.of_curve, self.bc_of, self.zhat = [], [], [], []
        self.near = torch.full((n,), -1, device=dev)
        first = n
        for k, cv in enumerate(self.curves):
            cc = self._cp_curve(cv, self.x)
            d = self.x - cc
            dist = torch.sqrt(_dot(d, d))
            self.near[dist < 2.0 * self.r] = k
            tw = (dist <= self.r).nonzero()[:, 0]
            of = torch.full((n,), -1, device=dev)
            of[tw] = first + torch.arange(tw.numel(), device=dev)
            first += tw.numel()
            z = self.cp - cc
            tiny = (torch.sqrt(_dot(z, z)) < 0.1 * self.h * self.h).nonzero()[:, 0]
            if tiny.numel():  # on the curve: the side of the first stencil node that is not
                nodes = self._stencil(self.cp[tiny])[0]
                zz = z[nodes.clamp(min=0)]
                good = (nodes >= 0) & (torch.sqrt(_dot(zz, zz)) >= 0.1 * self.h * self.h)
                pick = good.double().argmax(1)
                z = z.clone()
                z[tiny] = torch.where(good.any(1)[:, None], zz[torch.arange(tiny.numel(), device=dev), pick], torch.zeros_like(zz[:, 0]))
            self.twin.append(tw)
            self.of_curve.append(torch.full_like(tw, k))
            self.bc_of.append(of)
            self.zhat.append(z)
        self.twin = torch.cat(self.twin) if self.curves else torch.zeros(0, dtype=torch.long, device=dev)
        self.of_curve = torch.cat(self.of_curve) if self.curves else self.twin
        self.N = first
        o = [[-1, 0, 0], [1, 0, 0], [0, -1, 0], [0, 1, 0], [0, 0, -1], [0, 0, 1]][:2 * self.dim]
        self.fd = self._find(self.ijk[:, None, :] + torch.tensor(o, device=dev))
        for k in range(len(self.curves)):
            rows = (self.near == k).nonzero()[:, 0]
            self.fd[rows] = self._flip(k, self.zhat[k][rows], self.fd[rows])
        # boundary rows: the diagonal one, and for second order the mirror point's stencil
        self.brow, self.bcol, self.bval = [], [], []
        for k, cv in enumerate(self.curves):
            if self.bc != DIR2:
                continue
            tw = self.twin[self.of_curve == k]
            rows = self.bc_of[k][tw]
            y = 2.0 * self._cp_curve(cv, self.x[tw]) - self.x[tw]
            nodes, w = self._stencil(_cp_surface(self.kind, y))
            other = _dot(self.zhat[k][tw][:, None, :], self.zhat[k][nodes]) < 0.0
            twins = self.bc_of[k][nodes]
            cols = torch.where(other | (twins < 0), nodes, twins)
            self.brow.append(rows[:, None].expand_as(cols).reshape(-1))
            self.bcol.append(cols.reshape(-1))
            self.bval.append(w.reshape(-1))

    def _flip(self, k, dstar, nodes):
        """Nodes across curve k give way to their boundary twins."""
        at = nodes.clamp(min=0)
        tw = self.bc_of[k][at]
        return torch.where((nodes >= 0) & (_dot(dstar[:, None, :], self.zhat[k][at]) < 0.0) & (tw >= 0), tw, nodes)

    def rows_of_E(self, a, b):
        nodes, w = self._stencil(self.cp[a:b])
        near = self.near[a:b]
        for k in range(len(self.curves)):
            at = (near == k).nonzero()[:, 0]
            if at.numel():
                nodes[at] = self._flip(k, self.zhat[k][a:b][at], nodes[at])
        return nodes, w

    def _chunks(self, nrhs):
        step = max(1024, int(6e7 / (self.np1 ** self.dim * nrhs)))
        return [(a, min(self.n, a + step)) for a in range(0, self.n, step)]

    def extend(self, u):
        e = torch.empty_like(u)
        e[self.n:] = u[self.n:]
        for a, b in self._chunks(u.shape[1]):
            nodes, w = self.rows_of_E(a, b)
            ui = u[a:b]
            e[a:b] = ui + (w[:, :, None] * (u[nodes] - ui[:, None, :])).sum(1)
        return e

    def apply(self, m, n, u):
        e = self.extend(u)
        v = torch.empty_like(u)
        acc = torch.zeros_like(u[:self.n])
        for k in range(2 * self.dim):
            j = self.fd[:, k]
            acc += torch.where((j >= 0)[:, None], e[j.clamp(min=0)] - u[:self.n], -u[:self.n])
        v[:self.n] = m * u[:self.n] + n / self.h ** 2 * acc
        v[self.n:] = u[self.n:]
        for r, c, w in zip(self.brow, self.bcol, self.bval):
            v.index_add_(0, r, w[:, None] * u[c])
        return v

    def transpose(self, m, n, lam):
        s = n / self.h ** 2
        y = torch.zeros_like(lam)
        y[:self.n] = (m - 2 * self.dim * s) * lam[:self.n]
        y[self.n:] = lam[self.n:]
        b = torch.zeros_like(lam)
        for k in range(2 * self.dim):
            j = self.fd[:, k]
            ok = j >= 0
            b.index_add_(0, j[ok], s * lam[:self.n][ok])
        y[self.n:] += b[self.n:]
        for a, c in self._chunks(lam.shape[1]):
            nodes, w = self.rows_of_E(a, c)
            y.index_add_(0, nodes.reshape(-1), (w[:, :, None] * b[a:c, None, :]).reshape(-1, lam.shape[1]))
        for r, c, w in zip(self.brow, self.bcol, self.bval):
            y.index_add_(0, c, w[:, None] * lam[r])
        return y

    def matrices(self):
        """E and F with A = m I + n (F E - 2 dim / h^2) on PDE rows; B the boundary rows."""
        dev, N, one = self.dev, self.N, torch.ones
        r, c, v = [], [], []
        for a, b in self._chunks(1):
            nodes, w = self.rows_of_E(a, b)
            r.append(torch.arange(a, b, device=dev)[:, None].expand_as(nodes).reshape(-1))
            c.append(nodes.reshape(-1))
            v.append(w.reshape(-1))
        bc = torch.arange(self.n, N, device=dev)
        E = self._sparse(r + [bc], c + [bc], v + [one(N - self.n, dtype=torch.float64, device=dev)])
        rows = torch.arange(self.n, device=dev)[:, None].expand_as(self.fd)
        ok = self.fd >= 0
        F = self._sparse([rows[ok]], [self.fd[ok]], [torch.full((int(ok.sum()),), 1 / self.h ** 2, dtype=torch.float64, device=dev)])
        B = self._sparse([bc] + self.brow, [bc] + self.bcol, [one(N - self.n, dtype=torch.float64, device=dev)] + self.bval)
        return E, F, B

    def _sparse(self, r, c, v):
        i = torch.stack([torch.cat(r), torch.cat(c)])
        return torch.sparse_coo_tensor(i, torch.cat(v), (self.N, self.N)).coalesce()

    def solver(self, m, n):
        """x -> A^-1 x and A^-T x to rounding, by BiCGSTAB with restarts on the assembled factors."""
        E, F, B = self.matrices()
        pde = (torch.arange(self.N, device=self.dev) < self.n).double()[:, None]
        d = pde * (m - 2 * self.dim * n / self.h ** 2)
        diag = d + (1 - pde)
        fwd, bwd = [M.to_sparse_csr() for M in (E, F, B)], [M.t().coalesce().to_sparse_csr() for M in (E, F, B)]

        def A(x):
            return d * x + n * (fwd[1] @ (fwd[0] @ x)) + fwd[2] @ x

        def At(x):
            return d * x + n * (bwd[0] @ (bwd[1] @ x)) + bwd[2] @ x

        if self.N <= 12000:  # the circle: assembled and solved directly, refined once
            full = A(torch.eye(self.N, dtype=torch.float64, device=self.dev))
            lu, piv = torch.linalg.lu_factor(full)

            def direct(f, adjoint=False, x0=None):
                x = torch.linalg.lu_solve(lu, piv, f, adjoint=adjoint)
                return x + torch.linalg.lu_solve(lu, piv, f - (At(x) if adjoint else A(x)), adjoint=adjoint)

            return direct

        def solve(f, adjoint=False, x0=None):
            # row-scaled A, or its transpose by right preconditioning
            op = (lambda y: At(y / diag)) if adjoint else (lambda y: A(y) / diag)
            rhs = f if adjoint else f / diag
            y = torch.zeros_like(f) if x0 is None else x0.clone()
            fn = rhs.norm(dim=0)
            best, keep = None, y
            for attempt in range(12):
                r = rhs - op(y)
                rel = float((r.norm(dim=0) / fn.clamp(min=1e-300)).max())
                if best is None or rel < best:
                    gained = best is None or rel < 0.5 * best
                    best, keep = rel, y.clone()
                    if rel < 2e-16 or not gained:
                        break
                else:
                    break
                y = self._bicgstab(op, y, r, fn)
            return keep / diag if adjoint else keep

        return solve

    @staticmethod
    def _bicgstab(op, y, r, fn, most=6000):
        g = torch.Generator(device=r.device)
        g.manual_seed(5)
        rh = r.norm(dim=0) / math.sqrt(r.shape[0]) * torch.randn(r.shape, generator=g, dtype=r.dtype, device=r.device)
        start = r.norm(dim=0)
        p, v = torch.zeros_like(r), torch.zeros_like(r)
        rho = al = om = torch.ones_like(fn)
        live = start > 0
        tiny = 1e-300
        for it in range(most):
            rho1 = (rh * r).sum(0)
            beta = rho1 / torch.where(rho.abs() > tiny, rho, torch.ones_like(rho)) * (al / torch.where(om.abs() > tiny, om, torch.ones_like(om)))
            p = r + torch.where(live, beta, torch.zeros_like(beta)) * (p - om * v)
            v = op(p)
            den = (rh * v).sum(0)
            al = torch.where(live & (den.abs() > tiny), rho1 / torch.where(den.abs() > tiny, den, torch.ones_like(den)), torch.zeros_like(den))
            s = r - al * v
            t = op(s)
            tt = (t * t).sum(0)
            om = torch.where(live & (tt > tiny), (t * s).sum(0) / torch.where(tt > tiny, tt, torch.ones_like(tt)), torch.zeros_like(tt))
            y = y + torch.where(live, al, torch.zeros_like(al)) * p + om * s
            r = torch.where(live, s - om * t, r)
            rho = rho1
            if it % 20 == 19:
                rn = r.norm(dim=0)
                live = live & (rn > 1e-11 * start) & (rn > 1e-17 * fn) & torch.isfinite(rn)
                if not bool(live.any()):
                    break
        return torch.where(torch.isfinite(y), y, torch.zeros_like(y))

    def bc_data(self, case, samples):
        """c_alpha g_alpha from the curves' samples: periodic linear interpolation at the angle of cp_C, and
        its transpose (a dense matrix)."""
        G = torch.zeros((self.N - self.n, samples), dtype=torch.float64, device=self.dev)
        off = 0
        for k, (cv, ns) in enumerate(zip(self.curves, _samples(case))):
            at = (self.of_curve == k).nonzero()[:, 0]
            q = self._cp_curve(cv, self.x[self.twin[at]]) - torch.tensor(cv.p, dtype=torch.float64, device=self.dev)
            ref = torch.tensor(cv.ref, dtype=torch.float64, device=self.dev)
            e2 = torch.linalg.cross(torch.tensor(cv.nu, dtype=torch.float64, device=self.dev), ref)
            ang = torch.atan2(q @ e2, q @ ref) if cv.kind == 2 else torch.zeros(at.numel(), dtype=torch.float64, device=self.dev)
            sp = torch.remainder(ang, 2 * math.pi) / (2 * math.pi) * ns
            i0 = torch.floor(sp)
            fr = sp - i0
            i0 = i0.long() % ns
            G.index_put_((at, off + i0), 1.0 - fr, accumulate=True)
            G.index_put_((at, off + (i0 + 1) % ns), fr, accumulate=True)
            off += ns
        return G * (2.0 if self.bc == DIR2 else 1.0)


def exact(case, seed):
    n = _rows(case)
    if case["shape"] == "bumpy" or n * case["nrhs"] > 1.5e8:
        return None  # Newton projections of tens of millions of nodes, or too much to do in 64 bits
    if case["op"] in ("solve", "gradient", "heat", "steps") and (n > 6e5 or n * case["nrhs"] > 1.2e7):
        return None
    S = _System(case)
    z = _inputs(case, seed, S.cp, S.twin)
    col = (lambda t: t.double()[:, None] if t.dim() == 1 else t.double())  # noqa: E731
    flat = (lambda t: t[:, 0] if case["nrhs"] == 1 else t)  # noqa: E731
    op = case["op"]
    if op in ("apply", "transpose"):
        return flat(getattr(S, op)(0.0, 1.0, col(z["u"])))
    if op == "fields":
        return _exact_fields(S, z["u"])
    tot = sum(_samples(case))
    if op == "solve":
        f = torch.cat([col(z["s"]), S.bc_data(case, tot) @ col(z["samples"])])
        return flat(S.solver(0.0, 1.0)(f))
    if op == "heat":
        f = torch.cat([torch.zeros((S.n, 1), dtype=torch.float64, device=S.dev), S.bc_data(case, tot) @ col(z["samples"])])
        return flat(S.solver(1.0, -S.h)(f))
    if op == "steps":
        u, solve = col(z["u"]), S.solver(1.0, -0.5 * S.h)
        c = 2.0 if S.bc == DIR2 else 1.0
        for _ in range(case["steps"]):
            u = solve(torch.cat([S.apply(1.0, 0.5 * S.h, u)[:S.n], c * z["g"][:, None]]), x0=u)
        return u[:, 0]
    G, solve = S.bc_data(case, tot), S.solver(0.0, 1.0)
    u = solve(torch.cat([col(z["s"]), G @ col(z["samples"])]))
    lam = solve(u - col(z["target"]), adjoint=True)
    return u[:, 0], lam[:S.n, 0], (G.t() @ lam[S.n:])[:, 0]


def _exact_fields(S, u):
    e = S.extend(u[:, None])[:, 0]
    at = torch.cat([torch.arange(S.n, device=S.dev), S.twin])
    own = torch.arange(S.n, device=S.dev)

    def side(f, k, d=None):
        j = torch.where(S.fd[:, k] >= 0, S.fd[:, k], own)
        return f[j] if d is None else f[j, d]

    g = torch.zeros((S.n, 3), dtype=torch.float64, device=S.dev)
    for d in range(S.dim):
        g[:, d] = (side(e, 2 * d + 1) - side(e, 2 * d)) / (2 * S.h)
    nrm = torch.sqrt(_dot(g, g))[:, None]
    X = torch.where(nrm > 0, -g / nrm, torch.zeros_like(g))[at]
    Xe = S.extend(X)
    b = torch.zeros(S.n, dtype=torch.float64, device=S.dev)
    for d in range(S.dim):
        b += (side(Xe, 2 * d + 1, d) - side(Xe, 2 * d, d)) / (2 * S.h)
    return X, b
