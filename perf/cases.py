"""The calls whose speed is measured: whole MRCM-OS steps, new-permeability
passes and gradients through the public front end (``solver.MRCM`` and
``solver.mrcm_solve``), on the sizes and options this repository's workloads,
tests and benchmark use.

listed() names the cases, draw(rng) gives more of the same ranges,
prepare(case, seed) makes the inputs and the handle, run(state) is one pass,
work(case) counts what a pass cannot do without, and exact(case, seed) is the
same result from a dense 64-bit torch computation that shares no code with
the library (dense Cholesky per box, dense interface solve; gradients by
torch's own differentiation of it).
"""
import functools
import math
import random
from types import SimpleNamespace

import numpy as np
import torch

from paper_2404_13811_gb300 import inputs as I
from paper_2404_13811_gb300 import solver as S

NEUMANN, DIRICHLET = 0, 1


def _case(name, **kw):
    c = dict(kind="step", nx=64, ny=64, nz=1, sx=16, sy=16, sz=1, overlap=2, space=1, alpha_basis=1.0, steps=4,
             precision="mixed", particular="omega", field="lognormal", variance=4.0, contrast=1e4, bc="left_right", source="none",
             members=1)
    c.update(kw)
    c["name"] = name
    return c


def listed():
    return [
        # the smallest whole step in use: 16 subdomains, quarter five spot in a closed box, P0 spaces, a separate
        # smoothing factor (alpha_basis differs); what counts is latency and launches
        _case("q5_64_p0", nx=64, ny=64, space=0, alpha_basis=1e-2, bc="noflow", source="q5"),
        # the benchmark's step: 512 x 512 channels of contrast 1e4, 1024 subdomains, replayed as one graph
        _case("channel_512", nx=512, ny=512, overlap=4, steps=8, field="workload"),
        # the same step in the 64-bit form, the library's most exact setting
        _case("channel_512_fp64", nx=512, ny=512, overlap=4, steps=8, field="workload", precision="fp64"),
        # a grid as reservoirs have them: not square, odd subdomains (box lines of 18 and 21 cells), sources
        _case("ragged_225x192", nx=225, ny=192, sx=15, sy=12, overlap=3, steps=3, variance=2.0, source="random"),
        # the particular problem on the oversampled box (the variant without a second factor)
        _case("hat_256", nx=256, ny=256, overlap=4, steps=4, field="channel", contrast=1e3, variance=1.0,
              particular="hat"),
        # one sample of a Monte Carlo or inversion loop: a new permeability from host memory, the eager step (its
        # first solve tunes itself), pressure and velocities back on the host
        _case("new_k_256", kind="new_k", nx=256, ny=256, overlap=4, steps=4),
        # one iteration of a gradient-based inversion: forward and reverse pass with respect to log K
        _case("gradient_256", kind="gradient", nx=256, ny=256, overlap=4, steps=6, source="sinks"),
        # an ensemble of uneven members in one handle, one launch per kernel over all of them
        _case("ensemble_24", kind="ensemble", nx=128, ny=512, overlap=4, members=24),
        # 3D with linear interface spaces, planes of 80 cells and sources
        _case("block3d_48x36x40_p1", nx=48, ny=36, nz=40, sx=8, sy=6, sz=8, overlap=1, steps=2, variance=2.0,
              source="random"),
        # the 3D workload: 60 x 220 x 85 cells, channels of contrast 1e6 over log-normal layers
        _case("layered3d_full", nx=60, ny=220, nz=85, sx=10, sy=10, sz=5, space=0, field="workload"),
        # a part of it in the 64-bit form
        _case("layered3d_30x40x20_fp64", nx=30, ny=40, nz=20, sx=10, sy=10, sz=5, space=0, field="workload",
              precision="fp64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["2d", "2d", "2d", "2d", "new_k", "gradient", "ensemble", "3d", "3d", "layered"])
    c = _case("")
    del c["name"]
    c["precision"] = rng.choice(["mixed", "mixed", "fp64"])
    c["steps"] = rng.randint(1, 8)
    if kind in ("3d", "layered"):
        (c["sx"], c["sy"], c["sz"]), c["overlap"] = rng.choice(
            [((10, 10, 5), 2), ((8, 6, 8), 1), ((8, 8, 6), 2), ((6, 8, 5), 1), ((9, 7, 5), 2), ((7, 9, 6), 1)])
        top = 4 if c["precision"] == "fp64" else 6
        c["nx"], c["ny"], c["nz"] = (c[s] * _log_int(rng, 2, top) for s in ("sx", "sy", "sz"))
        c["steps"] = rng.randint(1, 4)
        c["variance"] = rng.uniform(1.0, 4.0)
        c["space"] = rng.choice([0, 1])
        c["source"] = rng.choice(["none", "random"])
        if kind == "layered":
            c.update(field="layered", space=0, source="none", variance=5.0, contrast=1e3)
        return c
    c["sx"], c["sy"] = rng.randint(8, 16), rng.randint(8, 16)
    c["overlap"] = rng.randint(1, min(4, (min(c["sx"], c["sy"]) - 1) // 2))
    blocks = 16 if kind == "gradient" else 32
    c["nx"], c["ny"] = c["sx"] * _log_int(rng, 3, blocks), c["sy"] * _log_int(rng, 3, blocks)
    c["space"] = rng.choice([0, 1, 1])
    c["variance"] = rng.uniform(2.0, 6.0)
    c["source"] = rng.choice(["none", "random"])
    if kind == "ensemble":
        c.update(kind="ensemble", sx=16, sy=16, nx=128, ny=rng.choice([256, 384, 512]), members=rng.randint(2, 24),
                 overlap=rng.randint(2, 4), steps=rng.randint(1, 4), source="none", variance=4.0)
        return c
    if kind in ("new_k", "gradient"):
        c["kind"] = kind
        c["source"] = "sinks" if kind == "gradient" else "none"
        return c
    c["alpha_basis"] = rng.choice([1.0, 1.0, 1.0, 0.05])
    c["particular"] = rng.choice(["omega", "omega", "omega", "hat"])
    if rng.random() < 0.3:
        c.update(field="channel", variance=1.0, contrast=1e3)
    if rng.random() < 0.25:
        c.update(bc="noflow", source="q5", field="lognormal")
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _dims(case):
    d = 3 if case["nz"] > 1 else 2
    return d, (case["nx"], case["ny"], case["nz"])[:d], (case["sx"], case["sy"], case["sz"])[:d]


def _gaussian(n, h, variance, length, gen):
    """Zero-mean Gaussian field of covariance variance exp(-r / length), circulant embedding on twice the grid;
    shape n[::-1], on the GPU."""
    r2 = 0.0
    for a, k in enumerate(n):
        x = torch.arange(2 * k, device="cuda", dtype=torch.float64)
        x = torch.minimum(x, 2 * k - x) * h[a]
        r2 = r2 + (x * x).reshape([-1 if b == a else 1 for b in reversed(range(len(n)))])
    lam = torch.fft.fftn(variance * torch.exp(-torch.sqrt(r2) / length)).real.clamp_(min=0.0)
    xi = torch.complex(torch.randn(lam.shape, generator=gen, device="cuda", dtype=torch.float64),
                       torch.randn(lam.shape, generator=gen, device="cuda", dtype=torch.float64))
    y = torch.fft.fftn(torch.sqrt(lam / lam.numel()) * xi).real
    return y[tuple(slice(0, k) for k in reversed(n))].contiguous()


def _channels(n, rng):
    """Mask of sinusoidal channels along x, 4 to 8 cells wide, a quarter of the area (in 3D each a few layers
    thick); shape n[::-1]."""
    nx, ny = n[0], n[1]
    nz = n[2] if len(n) == 3 else 1
    mask = np.zeros((nz, ny, nx), dtype=bool)
    x, y = np.arange(nx) + 0.5, np.arange(ny) + 0.5
    for _ in range(400):
        if mask.mean() >= 0.25:
            break
        mid = rng.uniform(0, ny) + rng.uniform(0.05, 0.25) * ny * np.sin(
            2 * math.pi * x / (rng.uniform(0.5, 1.5) * nx) + rng.uniform(0, 2 * math.pi))
        band = np.abs(y[:, None] - mid[None, :]) < 0.5 * rng.uniform(4.0, 8.0)
        z0 = rng.integers(0, nz)
        mask[z0:z0 + (int(rng.integers(2, 6)) if nz > 1 else 1)] |= band[None]
    return mask if len(n) == 3 else mask[0]


@functools.lru_cache(maxsize=None)
def _workload_field(n):
    """log K of the repository's channel (2D, contrast 1e4) or layered (3D, contrast 1e6) workload."""
    if len(n) == 2:
        return np.log(I.config_channel2d(n=n[0]).problem.K)
    return np.log(I.config_layered3d(n=n, n_upper=max(1, (n[2] * 35) // 85)).problem.K)


def _problem(case, n, sub, seed, variance=None):
    """One problem on the host: K and f as numpy arrays, boundary data (and, for gradients, the sink cells)."""
    d = len(n)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.default_rng(seed)
    cubes = d == 3 and case["field"] != "lognormal"
    h = (1.0 / 60,) * 3 if cubes else tuple(1.0 / k for k in n)
    variance = case["variance"] if variance is None else variance
    if case["field"] == "workload":
        # the workload's own field, each seed with its own fluctuations of 10 % on it
        K = np.exp(_workload_field(n) + _gaussian(n, h, 0.01, 0.1 * n[0] * h[0], gen).cpu().numpy())
    else:
        y = _gaussian(n, h, variance, 0.1 * n[0] * h[0] if cubes else 0.1 if d == 2 else 0.2, gen)
        K = torch.exp(y).cpu().numpy()
    if case["field"] == "channel":
        K = K * np.where(_channels(n, rng), case["contrast"], 1.0)
    elif case["field"] == "layered":
        up = max(1, (n[2] * 35) // 85)
        low = (n[0], n[1], n[2] - up)
        ylow = torch.exp(_gaussian(low, h, 1.0, 0.1 * n[0] * h[0], gen)).cpu().numpy()
        K[up:] = ylow * np.where(_channels(low, rng), case["contrast"], 1.0)
    f = np.zeros(n[::-1])
    vol = float(np.prod(h))
    sinks = []
    if case["source"] == "q5":
        f.flat[0], f.flat[-1] = 1.0 / vol, -1.0 / vol
    elif case["source"] == "random":
        f = rng.standard_normal(n[::-1])
    elif case["source"] == "sinks":
        while len(sinks) < 8:
            c = tuple(int(rng.integers(0, n[a])) for a in range(d))
            if c not in sinks and all(2 <= c[a] % sub[a] < sub[a] - 2 for a in range(d)):
                sinks.append(c)
                f[c[::-1]] = -1.0 / 8.0 / vol
    kind, val = [NEUMANN] * (2 * d), [0.0] * (2 * d)
    if case["bc"] == "left_right":
        kind[0] = kind[1] = DIRICHLET
        val[0] = 1.0
    return SimpleNamespace(dim=d, n=n, h=h, K=np.ascontiguousarray(K), f=f, bc_kind=tuple(kind), bc_value=tuple(val),
                           sinks=[c[0] + n[0] * c[1] for c in sinks],
                           target=rng.standard_normal((len(sinks), 2 * d)))


def _members(case):
    """(grid, overlap, variance) of the members of an ensemble: 16 round(n / 16) with n log-uniform between nx and
    ny, each its own variance and overlap, by the sizes alone."""
    rng = random.Random(404 + case["members"] + case["ny"])
    out = []
    for _ in range(case["members"]):
        k = max(32, 16 * round(math.exp(rng.uniform(math.log(case["nx"]), math.log(case["ny"]))) / 16))
        out.append(((k, k), rng.randint(2, case["overlap"]), rng.uniform(2.0, 6.0)))
    return out


def _problems(case, seed):
    d, n, sub = _dims(case)
    if case["kind"] != "ensemble":
        return [_problem(case, n, sub, seed)], [SimpleNamespace(sub=sub, overlap=case["overlap"])]
    ms = _members(case)
    return ([_problem(case, m[0], (16, 16), seed * 1000 + i, m[2]) for i, m in enumerate(ms)],
            [SimpleNamespace(sub=(16, 16), overlap=m[1]) for m in ms])


def prepare(case, seed):
    probs, parts = _problems(case, seed)
    many = case["kind"] == "ensemble"
    handle = S.MRCM(probs if many else probs[0], parts if many else parts[0], space=case["space"],
                    alpha_basis=case["alpha_basis"], alpha_smooth=1.0, precision=case["precision"],
                    particular=case["particular"])
    st = {"handle": handle, "case": case}
    if case["kind"] == "new_k":
        st["logk"] = torch.from_numpy(np.log(probs[0].K).reshape(-1)).pin_memory()
    elif case["kind"] == "gradient":
        st["logk"] = torch.from_numpy(np.log(probs[0].K).reshape(-1)).cuda()
        st["sinks"] = torch.tensor(probs[0].sinks, device="cuda")
        st["target"] = torch.from_numpy(probs[0].target).cuda()
    return st


def run(state):
    case, h = state["case"], state["handle"]
    if case["kind"] == "new_k":
        h.set_permeability(state["logk"], log=True)
        h.run(case["steps"])
        return h.fluxes()
    if case["kind"] == "gradient":
        logk = state["logk"].detach().requires_grad_(True)
        p, u = S.mrcm_solve(h, logk, case["steps"])
        loss = ((u[state["sinks"]] - state["target"]) ** 2).sum()
        grad, = torch.autograd.grad(loss, logk)
        return {"p": p.detach(), "u": u.detach(), "grad": grad}
    h.run(case["steps"], graph=True)
    if case["kind"] == "ensemble":
        return [h.fluxes(m, device=True) for m in range(case["members"])]
    return h.state()


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Bytes: K and f once, p and u once (a gradient more where there is one).  Flops: n b^2 for each block
    factor of n cells and band b, 4 n b for each solve, 2 m^3 for each interface layer of m unknowns; the basis
    and particular problems, the smoothing solves, and in a gradient one more solve for each of them."""
    d, n, sub = _dims(case)
    members = _members(case) if case["kind"] == "ensemble" else [(n, case["overlap"], 0.0)]
    npsi = 1 if case["space"] == 0 else d
    flops = nbytes = 0.0
    for n, ov, _ in members:
        cells = math.prod(n)
        nbytes += 8.0 * cells * (3 + 2 * d + (1 if case["kind"] == "gradient" else 0))
        M = [n[a] // sub[a] for a in range(d)]
        boxes = {(): 1}
        for a in range(d):
            new = {}
            for key, k in boxes.items():
                for i in range(M[a]):
                    e = (min(n[a], (i + 1) * sub[a] + ov) - max(0, i * sub[a] - ov), (i > 0) + (i < M[a] - 1))
                    new[key + (e,)] = new.get(key + (e,), 0) + k
            boxes = new
        unknowns = 0
        for key, k in boxes.items():
            nc = math.prod(e[0] for e in key)
            b = nc // max(e[0] for e in key)
            rhs = npsi * sum(e[1] for e in key)
            unknowns += k * rhs
            again = 2 if case["kind"] == "gradient" else 1
            same = case["alpha_basis"] == 1.0
            flops += k * (nc * b * b * (1 if same else 2) + 4.0 * nc * b * (rhs + case["steps"]) * again)
            if case["particular"] == "hat":
                flops += k * 4.0 * nc * b * again
        if case["particular"] != "hat":
            nc = math.prod(sub)
            b = nc // max(sub)
            flops += math.prod(M) * (nc * b * b + 4.0 * nc * b)
        flops += M[-1] * 2.0 * (unknowns / M[-1]) ** 3
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# the same result from dense 64-bit linear algebra
# ---------------------------------------------------------------------------
def _dense(case, prob, part, K):
    """(p, u) of the method for the permeability tensor K [cells], differentiable in K."""
    dev = K.device
    d, n, h, sub, ov = prob.dim, prob.n, prob.h, part.sub, part.overlap
    npsi = 1 if case["space"] == 0 else d
    st = [math.prod(n[:a]) for a in range(d)]
    M = [n[a] // sub[a] for a in range(d)]
    ms = [math.prod(M[:a]) for a in range(d)]
    vol, ncells = math.prod(h), math.prod(n)
    area = [vol / h[a] for a in range(d)]
    f = torch.from_numpy(prob.f.reshape(-1)).to(dev) * vol
    cell = torch.arange(ncells, device=dev)
    T, hk, wh = [], [], []
    for a in range(d):
        last = (cell // st[a]) % n[a] == n[a] - 1
        kn = K[torch.where(last, cell, cell + st[a])]
        T.append(torch.where(last, torch.zeros_like(K), 2 * area[a] / h[a] * K * (kn / (K + kn))))
        hk.append(h[a] / (2 * K))
        wh.append(sub[a] * h[a] * 0.5 * (1 / K + 1 / kn))
    NS = 2 * d * npsi

    def psi(idx, ext, a):
        """The functions of a side normal to axis a at cell positions idx (one tensor an axis) of a box of ext."""
        cols = [torch.ones(len(idx[0]), device=dev, dtype=torch.float64)]
        if npsi > 1:
            cols += [2.0 * (idx[b].double() + 0.5) / ext[b] - 1.0 for b in range(d) if b != a]
        return torch.stack(cols, 1)

    class Boxes:
        """All boxes of one shape: indices, boundary faces, Cholesky factors."""

        def __init__(self, subs, lo, ext, off, alpha):
            self.subs, self.ext, self.off = subs, ext, off
            nc = math.prod(ext)
            loc = torch.arange(nc, device=dev)
            ls = [math.prod(ext[:a]) for a in range(d)]
            self.pos = [(loc // ls[a]) % ext[a] for a in range(d)]
            low = torch.tensor(lo, device=dev)
            self.g = sum((low[:, a:a + 1] + self.pos[a]) * st[a] for a in range(d))
            A = torch.zeros(len(subs), nc, nc, device=dev, dtype=torch.float64)
            diag = torch.zeros(len(subs), nc, device=dev, dtype=torch.float64)
            self.inner, self.side = [], []
            for a in range(d):
                L = loc[self.pos[a] < ext[a] - 1]
                R = L + ls[a]
                t = T[a][self.g[:, L]]
                diag = diag.index_add(1, L, t).index_add(1, R, t)
                A = A.index_put((torch.arange(len(subs), device=dev)[:, None], L, R), -t)
                A = A.index_put((torch.arange(len(subs), device=dev)[:, None], R, L), -t)
                self.inner.append((L, R, t))
                for s in (0, 1):
                    c = loc[self.pos[a] == (0 if s == 0 else ext[a] - 1)]
                    g = self.g[:, c]
                    phys = (low[:, a] + (0 if s == 0 else ext[a]) == (0 if s == 0 else n[a]))[:, None]
                    gf = torch.where(phys, g, g if s else g - st[a])
                    beta = torch.where(phys, torch.zeros_like(hk[a][g]), alpha * wh[a][gf])
                    tb = area[a] / (hk[a][g] + beta)
                    if prob.bc_kind[2 * a + s] == NEUMANN:
                        tb = torch.where(phys, torch.zeros_like(tb), tb)
                    diag = diag.index_add(1, c, tb)
                    self.side.append((c, phys, beta, tb))
            self.chol = torch.linalg.cholesky(A + torch.diag_embed(diag))
            om = [(self.pos[a] >= off[a]) & (self.pos[a] < off[a] + sub[a]) for a in range(d)]
            self.omega = loc[torch.stack(om).all(0)]
            self.gamma = []
            for sid in range(2 * d):
                at = off[sid // 2] + (sub[sid // 2] - 1 if sid & 1 else 0)
                self.gamma.append(self.omega[self.pos[sid // 2][self.omega] == at])

        def solve(self, b):
            return torch.cholesky_solve(b, self.chol)

        def rhs(self, lam, sources, k=1):
            b = torch.zeros(*self.g.shape, k, device=dev, dtype=torch.float64)
            if sources:
                b = b + f[self.g][..., None]
            for sid, (c, phys, beta, tb) in enumerate(self.side):
                v = torch.zeros(len(self.subs), len(c), k, device=dev, dtype=torch.float64)
                if sources and prob.bc_kind[sid] == DIRICHLET:
                    v = torch.where(phys[..., None], (tb * prob.bc_value[sid])[..., None], v)
                if lam is not None and lam[sid] is not None:
                    v = torch.where(phys[..., None], v, tb[..., None] * lam[sid])
                b = b.index_add(1, c, v)
            return b

        def velocities(self, p, lam, sources):
            """Outward velocities [box, cell, side, rhs]."""
            u = [torch.zeros_like(p) for _ in range(2 * d)]
            for a in range(d):
                L, R, t = self.inner[a]
                fl = t[..., None] * (p[:, L] - p[:, R]) / area[a]
                u[2 * a + 1] = u[2 * a + 1].index_add(1, L, fl)
                u[2 * a] = u[2 * a].index_add(1, R, -fl)
            for sid, (c, phys, beta, tb) in enumerate(self.side):
                r = torch.zeros_like(p[:, c])
                if sources and prob.bc_kind[sid] == DIRICHLET:
                    r = torch.where(phys[..., None], torch.full_like(r, prob.bc_value[sid]), r)
                if lam is not None and lam[sid] is not None:
                    r = torch.where(phys[..., None], r, lam[sid].expand_as(r))
                u[sid] = u[sid].index_add(1, c, tb[..., None] * (p[:, c] - r) / area[sid // 2])
            return torch.stack(u, 2)

    def group(hat, alpha, want=None):
        found = {}
        for s in range(math.prod(M)):
            m = [(s // ms[a]) % M[a] for a in range(d)]
            if want is not None and sum((m[a] & 1) << a for a in range(d)) != want:
                continue
            o = ov if hat else 0
            lo = tuple(max(0, m[a] * sub[a] - o) for a in range(d))
            ext = tuple(min(n[a], (m[a] + 1) * sub[a] + o) - lo[a] for a in range(d))
            off = tuple(m[a] * sub[a] - lo[a] for a in range(d))
            found.setdefault((ext, off), []).append((s, lo))
        return [Boxes([s for s, _ in v], [lo for _, lo in v], ext, off, alpha) for (ext, off), v in found.items()]

    nsub = math.prod(M)
    ncell_i = math.prod(sub)
    z = lambda *k: torch.zeros(*k, device=dev, dtype=torch.float64)  # noqa: E731
    parts = {"P": z(nsub, ncell_i, NS + 1), "U": z(nsub, ncell_i, 2 * d, NS + 1), "F": z(nsub, 2 * d, npsi, NS + 1),
             "Q": z(nsub, 2 * d, npsi, NS + 1)}
    glob = torch.zeros(nsub, ncell_i, device=dev, dtype=torch.long)

    def put(B, p, u, slots, pi_beta):
        """Restriction to Omega_i, flux and face-pressure moments of its sides."""
        at = (torch.tensor(B.subs, device=dev)[:, None], torch.tensor(slots, device=dev)[None, :])
        idx = torch.tensor(B.subs, device=dev)
        glob[idx] = B.g[:, B.omega]
        po, uo = p[:, B.omega], u[:, B.omega]
        parts["P"] = parts["P"].index_put(_ix(at, ncell_i), po.permute(0, 2, 1))
        parts["U"] = parts["U"].index_put(_ix2(at, ncell_i, 2 * d), uo.permute(0, 3, 1, 2))
        F, Q = [], []
        for sid in range(2 * d):
            a, c = sid // 2, B.gamma[sid]
            ps = psi([B.pos[b][c] - B.off[b] for b in range(d)], sub, a) * area[a]
            un = u[:, c, sid]
            if pi_beta:
                pi = B.side[sid][2][..., None] * un
            else:
                pi = p[:, c] - un * hk[a][B.g[:, c]][..., None]
            F.append(torch.einsum("fm,bfk->bmk", ps, un))
            Q.append(torch.einsum("fm,bfk->bmk", ps, pi))
        F, Q = torch.stack(F, 1), torch.stack(Q, 1)
        parts["F"] = parts["F"].index_put(_ix2(at, 2 * d, npsi), F.permute(0, 3, 1, 2))
        parts["Q"] = parts["Q"].index_put(_ix2(at, 2 * d, npsi), Q.permute(0, 3, 1, 2))

    def _ix(at, k):
        return at[0][..., None], torch.arange(k, device=dev)[None, None], at[1][..., None]

    def _ix2(at, k, m):
        return (at[0][..., None, None], torch.arange(k, device=dev)[None, None, :, None],
                torch.arange(m, device=dev)[None, None, None], at[1][..., None, None])

    hats = group(True, case["alpha_basis"])
    for B in hats:
        lam = []
        for sid, (c, phys, beta, tb) in enumerate(B.side):
            v = z(len(c), NS)
            v[:, sid * npsi:(sid + 1) * npsi] = psi([B.pos[b][c] for b in range(d)], B.ext, sid // 2)
            lam.append(v[None])
        p = B.solve(B.rhs(lam, False, NS))
        put(B, p, B.velocities(p, lam, False), list(range(NS)), False)
    for B in (hats if case["particular"] == "hat" else group(False, case["alpha_basis"])):
        p = B.solve(B.rhs(None, True))
        put(B, p, B.velocities(p, None, True), [NS], case["particular"] != "hat")

    # interface: unknown (s, side, m); the flux row of an edge sits at its lower subdomain's high side, the pressure
    # row at its upper subdomain's low side, an identity row where a side is on the boundary
    F, Q = parts["F"], parts["Q"]
    G, rhs = z(nsub * NS, nsub * NS), z(nsub * NS)
    active = z(nsub * NS)
    every = torch.arange(nsub, device=dev)
    for a in range(d):
        lo = every[(every // ms[a]) % M[a] < M[a] - 1]
        hi = lo + ms[a]
        for m in range(npsi):
            for mom, side, owner, sg in ((F, 2 * a + 1, lo, 1.0), (Q, 2 * a, hi, -1.0)):
                row = owner * NS + side * npsi + m
                for who, sid, w in ((lo, 2 * a + 1, 1.0), (hi, 2 * a, sg)):
                    cols = who[:, None] * NS + torch.arange(NS, device=dev)
                    G = G.index_put((row[:, None], cols), w * mom[who, sid, m, :NS])
                rhs = rhs.index_put((row,), -(mom[lo, 2 * a + 1, m, NS] + sg * mom[hi, 2 * a, m, NS]))
                active[row] = 1.0
    if all(k == NEUMANN for k in prob.bc_kind):
        # the constant: the first unknown is fixed in place of its (redundant) flux row
        first = int(torch.nonzero(active)[0])
        keep = torch.ones_like(rhs)
        keep[first] = 0.0
        G, rhs = G * keep[:, None], rhs * keep
        active[first] = 0.0
    G = G * active[:, None] + torch.diag(1.0 - active)
    r = 1.0 / G.detach().abs().amax(1)
    c = 1.0 / (G.detach() * r[:, None]).abs().amax(0)
    Ge = G * r[:, None] * c
    X = torch.linalg.solve(Ge, r * rhs)
    if not G.requires_grad:
        lu = torch.linalg.lu_factor(Ge)
        for _ in range(3):
            X = X + torch.linalg.lu_solve(*lu, (r * (rhs - G @ (c * X)))[:, None])[:, 0]
        del lu
    X = (c * X).reshape(nsub, NS)
    del G, Ge
    p = z(ncells).index_put((glob,), parts["P"][..., NS] + torch.einsum("sck,sk->sc", parts["P"][..., :NS], X))
    u = z(ncells, 2 * d).index_put((glob,), parts["U"][..., NS] + torch.einsum("scik,sk->sci", parts["U"][..., :NS], X))

    if case["steps"]:
        del hats
        colours = [group(True, 1.0, c) for c in range(1 << d)]
        for _ in range(case["steps"]):
            for boxes in colours:
                todo = []
                for B in boxes:
                    lam = []
                    for sid, (c, phys, beta, tb) in enumerate(B.side):
                        un = u[B.g[:, c], sid]
                        lam.append((-beta * un + p[B.g[:, c]] - un * hk[sid // 2][B.g[:, c]])[..., None])
                    x = B.solve(B.rhs(lam, True))
                    todo.append((B.g[:, B.omega], x[:, B.omega, 0], B.velocities(x, lam, True)[:, B.omega, :, 0]))
                for g, x, v in todo:
                    p, u = p.index_put((g,), x), u.index_put((g,), v)
    if all(k == NEUMANN for k in prob.bc_kind):
        p = p - p.mean()
    return p, u


def exact(case, seed):
    d, n, _ = _dims(case)
    if d == 3 and math.prod(n) > 100_000:
        return None  # thousands of dense factors of 1764 cells: more than about 20 seconds
    probs, parts = _problems(case, seed)
    if case["kind"] == "gradient":
        prob = probs[0]
        logk = torch.from_numpy(np.log(prob.K).reshape(-1)).cuda().requires_grad_(True)
        p, u = _dense(case, prob, parts[0], torch.exp(logk))
        loss = ((u[torch.tensor(prob.sinks, device="cuda")] - torch.from_numpy(prob.target).cuda()) ** 2).sum()
        grad, = torch.autograd.grad(loss, logk)
        return {"p": p.detach(), "u": u.detach(), "grad": grad}
    out = []
    with torch.no_grad():
        for i, (prob, part) in enumerate(zip(probs, parts)):
            # of an ensemble the first two members: each is a problem of its own
            out.append(_dense(case, prob, part, torch.from_numpy(prob.K.reshape(-1)).cuda()) if i < 2 else (None, None))
    return out if case["kind"] == "ensemble" else out[0]
