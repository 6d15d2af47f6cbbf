"""The work that is timed: calls through the public entry points, over the range of sizes they are used at.

A case is a dict of plain values.  `call` says which entry points a pass goes through:

  step     Plan.set_points, Plan.adjoint, Plan.forward: points that change from pass to pass
  solve    Plan.adjoint, Plan.forward on points set before: one iteration of a solver
  batch    Batch.set_points, Batch.adjoint, Batch.forward: many transforms, some with several right-hand sides
  energy   Plan.set_points, Plan.ewald_reciprocal: the reciprocal Ewald energy of a crystal
  forces   Plan.set_points, Plan.ewald_reciprocal_forces: the reciprocal part of a molecular-dynamics step
  real     ewald_real_space_forces: its real-space part

Forces that are computed in single precision are taken as such, as a mixed-precision integrator does.

The 64-bit values of exact() come from a gridding NFFT written in plain torch with a finer window (its error is far
below that of every plan here) and from a plain pair sum over cells.
"""
import math

import torch

from paper_2001_01583_gb300 import Batch, Plan
from paper_2001_01583_gb300.nfft import ewald_real_space_forces

EDGE = 4.0 / math.sqrt(3.0)   # edge of a fluorite cell, in units of the cation-anion distance


def _transform(name, call, N, M, m, window="kaiser_bessel", precision="fp32", clusters=0, std=0.0, sigma=2.0):
    c = dict(call=call, d=len(N), M=M, m=m, window=window, precision=precision, clusters=clusters, std=std, sigma=sigma)
    c.update({"N%d" % t: n for t, n in enumerate(N)})
    return dict(c, name=name) if name else c


def _batch(name, count, m_lo, m_hi, m_rhs, nrhs, m, draw_seed):
    c = dict(call="batch", count=count, m_lo=m_lo, m_hi=m_hi, m_rhs=m_rhs, nrhs=nrhs, m=m, draw_seed=draw_seed)
    return dict(c, name=name) if name else c


def _crystal(name, call, cells, N, m, alpha, precision="fp32"):
    c = dict(call=call, cells=cells, N=N, m=m, alpha=alpha, precision=precision)
    return dict(c, name=name) if name else c


def _pairs(name, cells, rcut, alpha):
    c = dict(call="real", cells=cells, rcut=rcut, alpha=alpha)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest calls: a short 1-D series in double precision, where launches and latency are all there is
        _transform("line_1d_fp64", "step", (256,), 1024, 6, "gaussian", "fp64"),
        # a 2-D image from scattered samples (non-Cartesian imaging), odd sizes
        _transform("image_2d", "step", (480, 362), 123457, 4),
        # few points on a fine grid: particles in a mostly empty box
        _transform("sparse_3d", "step", (64, 64, 64), 20000, 4),
        # the ordinary 3-D transform pair, points everywhere
        _transform("uniform_3d", "step", (64, 64, 64), 1000000, 4),
        # the same with clustered points (density peaks of a simulation)
        _transform("clustered_3d", "step", (64, 64, 64), 1000000, 4, clusters=32, std=0.02),
        # the same in double precision
        _transform("double_3d", "step", (64, 64, 64), 1000000, 4, precision="fp64"),
        # one iteration of a solver: fixed points, ragged grid, wider window
        _transform("ragged_solve_3d", "solve", (90, 128, 74), 777777, 5),
        # the largest: 256^3 modes and 3e7 clustered points at an accuracy of 1e-5
        _transform("largest_3d", "step", (256, 256, 256), 30000000, 3, clusters=64, std=0.01),
        # many small transforms of uneven size, and one point set with 16 right-hand sides
        _batch("batch_3d", 128, 1000, 100000, 200000, 16, 4, 0),
        # reciprocal Ewald energy of a fluorite crystal of 32^3 cells (393216 ions)
        _crystal("crystal_energy", "energy", 32, 128, 6, 0.6),
        # reciprocal forces of a molecular-dynamics step (96000 ions)
        _crystal("md_forces", "forces", 20, 64, 4, 0.6),
        # the real-space part of such a step (393216 ions, about 4000 partners each)
        _pairs("real_space_forces", 32, 10.0, 0.3),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _even(v):
    return max(2, 2 * int(round(v / 2)))


def draw(rng):
    call = rng.choice(["step"] * 5 + ["solve"] * 3 + ["batch", "energy", "forces", "real"])
    if call == "batch":
        return _batch(None, rng.randint(8, 128), 1000, int(_log(rng, 5000, 100000)), int(_log(rng, 5000, 200000)),
                      rng.randint(2, 16), rng.choice([3, 4, 5]), rng.randrange(1 << 20))
    if call in ("energy", "forces"):
        cells = rng.randint(6, 32 if call == "energy" else 24)
        return _crystal(None, call, cells, _even(_log(rng, 32, 128)), rng.choice([3, 4, 5, 6]),
                        round(rng.uniform(0.4, 0.9), 3), rng.choice(["fp32", "fp32", "fp32", "fp64"]))
    if call == "real":
        cells = rng.randint(6, 32)
        rcut = min(round(rng.uniform(4.0, 10.0), 2), round(0.32 * cells * EDGE, 2))
        return _pairs(None, cells, rcut, round(3.2 / rcut, 3))
    d = rng.choice([1, 2, 3, 3, 3, 3])
    precision = rng.choice(["fp32"] * 4 + ["fp64"])
    window = rng.choice(["kaiser_bessel"] * 4 + ["gaussian"])
    m = rng.randint(2, 6) if precision == "fp32" else rng.randint(4, 8)
    lo, hi = {1: (64, 65536), 2: (24, 1024), 3: (20, 150)}[d]
    base = _log(rng, lo, hi)
    N = tuple(_even(base * rng.uniform(0.75, 1.3)) for _ in range(d))
    # no more window cells than the largest listed case (double precision: than its listed case)
    cells = (2 * m + 2) ** d
    most = 6.0e9 / cells if precision == "fp32" else 5.0e8 / cells
    M = int(_log(rng, 1000, min(most, {1: 1e6, 2: 4e6, 3: 1e7}[d])))
    clusters, std = rng.choice([(0, 0.0), (0, 0.0), (32, 0.02), (64, round(_log(rng, 0.005, 0.1), 4))])
    return _transform(None, call, N, M, m, window, precision, clusters, std, rng.choice([2.0, 2.0, 2.0, 1.5]))


# ---------------------------------------------------------------------------
# inputs


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _points(M, d, clusters, std, g):
    if not clusters:
        return torch.rand((M, d), generator=g, dtype=torch.float64, device="cuda") - 0.5
    centres = torch.rand((clusters, d), generator=g, dtype=torch.float64, device="cuda") - 0.5
    which = torch.randint(0, clusters, (M,), generator=g, device="cuda")
    x = torch.randn((M, d), generator=g, dtype=torch.float64, device="cuda").mul_(std).add_(centres[which])
    return x.sub_(torch.floor(x + 0.5))


def _values(shape, dtype, g):
    real = torch.float64 if dtype == torch.complex128 else torch.float32
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), generator=g, dtype=real, device="cuda"))


def _dims(case):
    return tuple(case["N%d" % t] for t in range(case["d"]))


def _dtype(case):
    return torch.complex128 if case.get("precision") == "fp64" else torch.complex64


def _transform_inputs(case, seed):
    g = _generator(seed)
    x = _points(case["M"], case["d"], case["clusters"], case["std"], g)
    return x, _values((case["M"],), _dtype(case), g), _values(_dims(case), _dtype(case), g)


def _batch_items(case):
    g = torch.Generator()
    g.manual_seed(case["draw_seed"])
    u = torch.rand((case["count"], 2), generator=g, dtype=torch.float64)
    span = math.log(case["m_hi"] / case["m_lo"])
    items = [dict(N=(32 if float(a) < 0.5 else 64,) * 3, M=int(case["m_lo"] * math.exp(float(b) * span)), nrhs=1)
             for a, b in u]
    return items + [dict(N=(64, 64, 64), M=case["m_rhs"], nrhs=case["nrhs"])]


def _batch_inputs(case, seed):
    g = _generator(seed)
    xs, fs, hs = [], [], []
    for it in _batch_items(case):
        xs.append(_points(it["M"], 3, 0, 0.0, g))
        fs.append(_values((it["nrhs"], it["M"]), torch.complex64, g))
        hs.append(_values((it["nrhs"],) + it["N"], torch.complex64, g))
    return xs, fs, hs


def _ions(cells, seed):
    """Fluorite with thermal displacements: positions (units of the cation-anion distance), charges, box edge."""
    sites = [(0, 0, 0), (0, .5, .5), (.5, 0, .5), (.5, .5, 0)]
    sites += [(a, b, c) for a in (.25, .75) for b in (.25, .75) for c in (.25, .75)]
    sites = torch.tensor(sites, dtype=torch.float64, device="cuda")
    charge = torch.tensor([2.0] * 4 + [-1.0] * 8, dtype=torch.float64, device="cuda")
    k = torch.arange(cells, dtype=torch.float64, device="cuda")
    corner = torch.stack(torch.meshgrid(k, k, k, indexing="ij"), -1).reshape(-1, 1, 3)
    r = ((corner + sites) * EDGE).reshape(-1, 3)
    g = _generator(seed)
    r = r + 0.1 * torch.randn(r.shape, generator=g, dtype=torch.float64, device="cuda")
    # a program's atoms are not in lattice order
    order = torch.randperm(r.shape[0], generator=g, device="cuda")
    return r[order].contiguous(), charge.repeat(cells ** 3)[order].contiguous(), cells * EDGE


def prepare(case, seed):
    call = case["call"]
    if call in ("step", "solve"):
        x, f, fhat = _transform_inputs(case, seed)
        plan = Plan(_dims(case), case["M"], case["sigma"], case["m"], case["window"], case["precision"])
        if call == "solve":
            plan.set_points(x)
        return dict(call=call, plan=plan, x=x, f=f, fhat=fhat)
    if call == "batch":
        items = _batch_items(case)
        xs, fs, hs = _batch_inputs(case, seed)
        # the results side by side in one buffer per direction
        fhat = torch.empty(sum(h.numel() for h in hs), dtype=torch.complex64, device="cuda")
        f = torch.empty(sum(v.numel() for v in fs), dtype=torch.complex64, device="cuda")
        fhat_out = [b.view(h.shape) for b, h in zip(fhat.split([h.numel() for h in hs]), hs)]
        f_out = [b.view(v.shape) for b, v in zip(f.split([v.numel() for v in fs]), fs)]
        return dict(call=call, batch=Batch(items, "fp32", m=case["m"]), xs=xs, fs=fs, hs=hs, fhat=fhat, f=f,
                    fhat_out=fhat_out, f_out=f_out)
    r, q, L = _ions(case["cells"], seed)
    if call == "real":
        return dict(call=call, r=r, q=q, L=L, alpha=case["alpha"], rcut=case["rcut"])
    plan = Plan((case["N"],) * 3, r.shape[0], 2.0, case["m"], "kaiser_bessel", case["precision"])
    return dict(call=call, plan=plan, x=r / L - 0.5, q=q.to(_dtype(case)), L=L, alpha=case["alpha"])


def run(s):
    call = s["call"]
    if call in ("step", "solve"):
        if call == "step":
            s["plan"].set_points(s["x"])
        return s["plan"].adjoint(s["f"]), s["plan"].forward(s["fhat"])
    if call == "batch":
        s["batch"].set_points(s["xs"])
        s["batch"].adjoint(s["fs"], s["fhat_out"])
        s["batch"].forward(s["hs"], s["f_out"])
        return s["fhat"], s["f"]
    if call == "real":
        F, energy = ewald_real_space_forces(s["r"], s["q"], s["L"], s["alpha"], s["rcut"])
        return F.float(), energy
    s["plan"].set_points(s["x"])
    if call == "energy":
        return s["plan"].ewald_reciprocal(s["q"], s["L"], s["alpha"])
    F = s["plan"].ewald_reciprocal_forces(s["q"], s["L"], s["alpha"])
    return F.float() if s["q"].dtype == torch.complex64 else F


# ---------------------------------------------------------------------------
# what a pass cannot do without


def _pair_work(N, M, taps, sigma, nrhs, complex_bytes, points, adjoints=1, forwards=1):
    """Points and values read, results written; window cells (one complex multiply-add each) and the two FFTs."""
    NN = math.prod(N)
    n = math.prod(math.ceil(sigma * v) for v in N)
    passes = adjoints + forwards
    return dict(bytes=(8 * len(N) * M if points else 0) + passes * nrhs * complex_bytes * (M + NN),
                flops=passes * nrhs * (4.0 * M * taps ** len(N) + 5.0 * n * math.log2(n)))


def work(case):
    call = case["call"]
    if call in ("step", "solve"):
        taps = 2 * case["m"] + (2 if case["window"] == "gaussian" else 0)
        return _pair_work(_dims(case), case["M"], taps, case["sigma"], 1, 16 if case["precision"] == "fp64" else 8,
                          call == "step")
    if call == "batch":
        parts = [_pair_work(it["N"], it["M"], 2 * case["m"], 2.0, it["nrhs"], 8, True) for it in _batch_items(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    ions = 12 * case["cells"] ** 3
    if call == "real":
        pairs = ions * (4.0 / 3.0 * math.pi * case["rcut"] ** 3) * 12.0 / EDGE ** 3
        return dict(bytes=ions * (24 + 8 + 24), flops=40.0 * pairs)
    cb = 16 if case["precision"] == "fp64" else 8
    N, taps = (case["N"],) * 3, 2 * case["m"]
    if call == "energy":
        return dict(bytes=ions * (24 + cb), flops=_pair_work(N, ions, taps, 2.0, 1, cb, True, 1, 0)["flops"])
    return dict(bytes=ions * (24 + cb + 24), flops=_pair_work(N, ions, taps, 2.0, 1, cb, True, 1, 3)["flops"])


# ---------------------------------------------------------------------------
# the same in 64 bits


class _Fine:
    """A gridding NFFT in plain torch, 64 bits: twofold oversampling, Kaiser-Bessel window of cut-off m."""

    def __init__(self, x, N, m):
        self.x, self.N, self.m, self.b = x, N, m, 1.5 * math.pi
        self.n = [max(2 * v, 2 * m + 2) for v in N]
        self.chunk = max(1, (1 << 25) // (2 * m) ** len(N))
        self.scale = None
        for t, (v, n) in enumerate(zip(N, self.n)):
            k = torch.arange(-(v // 2), v // 2, dtype=torch.float64, device=x.device)
            arg = m * torch.sqrt(math.pi ** 2 * (2 - v / n) ** 2 - (2 * math.pi * k / n) ** 2)
            c = torch.special.i0e(arg) * torch.exp(arg - self._shape(t) * m)
            c = c.reshape([-1 if i == t else 1 for i in range(len(N))])
            self.scale = c if self.scale is None else self.scale * c
        self.modes = torch.meshgrid(*[torch.arange(-(v // 2), v // 2, device=x.device) % n for v, n in zip(N, self.n)],
                                    indexing="ij")

    def _shape(self, t):
        return math.pi * (2 - self.N[t] / self.n[t])

    def _chunks(self):
        d, taps = len(self.N), 2 * self.m
        for lo in range(0, self.x.shape[0], self.chunk):
            x = self.x[lo:lo + self.chunk]
            idx, w = None, None
            for t in range(d):
                u = self.n[t] * (x[:, t] - torch.floor(x[:, t] + 0.5))
                c = torch.floor(u)
                cell = c[:, None] + torch.arange(1 - self.m, self.m + 1, device=x.device)
                z2 = (self.m ** 2 - (u[:, None] - cell) ** 2).clamp_min(0.0)
                z, b = torch.sqrt(z2), self._shape(t)
                psi = torch.exp(b * (z - self.m)) * torch.where(z > 1e-12, -torch.expm1(-2 * b * z) / (2 * math.pi * z),
                                                                b / math.pi)
                i = cell.long() % self.n[t]
                idx = i if idx is None else (idx[:, :, None] * self.n[t] + i[:, None, :]).flatten(1)
                w = psi if w is None else (w[:, :, None] * psi[:, None, :]).flatten(1)
            yield lo, idx, w

    def adjoint(self, f):
        """f: (R, M) -> (R,) + N."""
        grids = torch.zeros((f.shape[0], math.prod(self.n), 2), dtype=torch.float64, device=f.device)
        f = torch.view_as_real(f.to(torch.complex128))
        for lo, idx, w in self._chunks():
            for r in range(f.shape[0]):
                v = f[r, lo:lo + w.shape[0]]
                grids[r].index_add_(0, idx.flatten(), (w[:, :, None] * v[:, None, :]).reshape(-1, 2))
        return torch.stack([torch.fft.fftn(torch.view_as_complex(g).reshape(self.n))[self.modes] / self.scale
                            for g in grids])

    def forward(self, fhat):
        """fhat: (R,) + N -> (R, M)."""
        out = torch.empty((fhat.shape[0], self.x.shape[0]), dtype=torch.complex128, device=fhat.device)
        grids = []
        for h in fhat:
            g = torch.zeros(self.n, dtype=torch.complex128, device=fhat.device)
            g[self.modes] = h.to(torch.complex128) / self.scale
            grids.append((torch.fft.ifftn(g) * float(math.prod(self.n))).flatten())
        for lo, idx, w in self._chunks():
            for r, g in enumerate(grids):
                out[r, lo:lo + w.shape[0]] = (g[idx] * w).sum(1)
        return out


def _fine(x, N, passes=1):
    """The finest window that takes a few seconds; None if none does."""
    for m in (10, 8, 6):
        if passes * x.shape[0] * (2 * m) ** len(N) <= 1.2e10:
            return _Fine(x, N, m)
    return None


def _pair_sum(r, q, L, alpha, rcut):
    """Real-space energy and forces, 64 bits: the ions of a cell against those of the cells around it."""
    nc = int(L / rcut)
    r = r - L * torch.floor(r / L)
    c = (r / (L / nc)).long().clamp_max(nc - 1)
    cell = (c[:, 0] * nc + c[:, 1]) * nc + c[:, 2]
    order = torch.argsort(cell)
    rs, qs = r[order], q[order]
    count = torch.bincount(cell, minlength=nc ** 3)
    end = torch.cumsum(count, 0).tolist()
    start = [0] + end[:-1]
    F, energy = torch.zeros_like(r), torch.zeros((), dtype=torch.float64, device=r.device)
    for a in range(nc ** 3):
        if end[a] == start[a]:
            continue
        ca = (a // (nc * nc), a // nc % nc, a % nc)
        near = sorted({((ca[0] + i) % nc * nc + (ca[1] + j) % nc) * nc + (ca[2] + k) % nc
                       for i in (-1, 0, 1) for j in (-1, 0, 1) for k in (-1, 0, 1)})
        rj = torch.cat([rs[start[b]:end[b]] for b in near])
        qj = torch.cat([qs[start[b]:end[b]] for b in near])
        for lo in range(start[a], end[a], 2048):
            hi = min(end[a], lo + 2048)
            d = [rs[lo:hi, None, t] - rj[None, :, t] for t in range(3)]
            d = [v - L * torch.round(v / L) for v in d]
            d2 = d[0] ** 2 + d[1] ** 2 + d[2] ** 2
            inside = (d2 < rcut * rcut) & (d2 > 0)
            d2 = torch.where(inside, d2, 1.0)
            dist = torch.sqrt(d2)
            e = torch.where(inside, torch.special.erfc(alpha * dist) / dist, 0.0) * qj
            g = torch.where(inside, 2 * alpha / math.sqrt(math.pi) * torch.exp(-alpha * alpha * d2), 0.0) * qj
            energy += 0.5 * (qs[lo:hi] * e.sum(1)).sum()
            g = (e + g) / d2
            F[order[lo:hi]] = torch.stack([(g * v).sum(1) for v in d], 1) * qs[lo:hi, None]
    return F, float(energy)


def exact(case, seed):
    call = case["call"]
    if call in ("step", "solve"):
        x, f, fhat = _transform_inputs(case, seed)
        fine = _fine(x, _dims(case))
        return None if fine is None else (fine.adjoint(f[None])[0], fine.forward(fhat[None])[0])
    if call == "batch":
        outs, vals = [], []
        for x, f, h in zip(*_batch_inputs(case, seed)):
            fine = _Fine(x, tuple(h.shape[1:]), 6)
            outs.append(fine.adjoint(f).flatten())
            vals.append(fine.forward(h).flatten())
        return torch.cat(outs), torch.cat(vals)
    r, q, L = _ions(case["cells"], seed)
    if call == "real":
        return _pair_sum(r, q, L, case["alpha"], case["rcut"])
    N = (case["N"],) * 3
    fine = _fine(r / L - 0.5, N, 1 if call == "energy" else 3)
    S = fine.adjoint(q[None].to(torch.complex128))[0]
    k = torch.meshgrid(*[torch.arange(-(v // 2), v // 2, dtype=torch.float64, device="cuda") for v in N], indexing="ij")
    k2 = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    w = torch.where(k2 > 0, torch.exp(-math.pi ** 2 * k2 / (case["alpha"] * L) ** 2) / k2.clamp_min(1.0), 0.0)
    if call == "energy":
        total = float((w * (S.real ** 2 + S.imag ** 2)).sum()) / (2 * math.pi * L)
        own = -case["alpha"] / math.sqrt(math.pi) * float((q * q).sum())
        return total + own, total, own
    modes = torch.stack([w * v * S for v in k])
    # the mode -N/2 has no partner in I_N: the sum over I_N is taken as it stands
    return 2.0 / L ** 2 * (q * fine.forward(modes).imag).T.contiguous()
