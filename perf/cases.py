"""Performance cases of the near-field, far-field and time-step entry points.

``listed()`` names the workloads a program that integrates an N-body box runs
call after call, from the smallest box of a batch to the 512^3 benchmark box;
``draw(rng)`` gives further cases of the same ranges.  ``prepare`` makes the
inputs and whatever the program keeps between calls (the derivatives tensor, a
captured graph, workspaces), ``run`` makes one call, ``work`` says what that
call cannot do without, and ``exact`` computes the same outputs in 64 bits with
plain torch.

Particles are about 64 per cell with a softening of 1/40 of the mean spacing,
as in ``workloads/recipes.py``; its clustered recipe (40 % uniform background,
60 % in Plummer spheres with Pareto member counts) is drawn here on the GPU.
"""
from __future__ import annotations

import math
import random

import torch

import paper_2110_11392_gb300 as nf
from paper_2110_11392_gb300 import _lib

DEV = "cuda"
F64 = torch.float64

# exact() is given up above this many ordered near-field pairs (about 10 s)
EXACT_PAIRS = 4e10
# pairs of the clustered recipe over those of a uniform box of the same size (1.5 at 128^3, 1.62 at 512^3)
CLUSTERED_PAIRS = 1.6


def listed():
    return [
        # the smallest box of a parameter scan or a unit test: launches and latency count
        dict(name="forces_4k", op="forces", N=4096, K=5, R=2, box=1.0, clustered=False),
        # a small uniform box, the plain configuration of the tests
        dict(name="forces_32k", op="forces", N=32768, K=8, R=2, box=1.0, clustered=False),
        # one training step of a field-level inference on a 64^3 box: autograd forward and backward
        dict(name="train_64c", op="train", N=64 ** 3, K=16, R=2, box=1.0, clustered=True),
        # the force call of a clustered 128^3 simulation
        dict(name="forces_128c", op="forces", N=128 ** 3, K=32, R=2, box=1.0, clustered=True),
        # the adjoint of a 256^3 box: the backward half of a large training step
        dict(name="adjoint_256c", op="adjoint", N=256 ** 3, K=64, R=2, box=1.0, clustered=True),
        # the benchmark box, forward: what a production run spends its time on
        dict(name="forces_512c", op="forces", N=512 ** 3, K=128, R=2, box=1.0, clustered=True),
        # forces with the friends-of-friends density of a group finder; ragged N, a grid and a box
        # side that are not powers of two
        dict(name="density_1m", op="density", N=1000003, K=25, R=2, box=3.7, clustered=True, b=0.2),
        # an ensemble of small boxes in one captured graph
        dict(name="batch_24", op="batch", boxes=24, n_lo=16 ** 3, n_hi=64 ** 3, sizes=4, clustered=True),
        # re-binning a large snapshot in Mpc/h coordinates (analysis codes sort without forces)
        dict(name="bin_30m", op="bin", N=30000001, K=101, box=500.0, clustered=False),
        # the far field of the 128^3 box at the paper's order
        dict(name="far_128c", op="far", N=128 ** 3, K=32, R=2, box=1.0, clustered=True, p=8),
        # the paper's Ewald test: 65536 random particles, 11^3 cells, order 8, near + far
        dict(name="total_65k", op="total", N=65536, K=11, R=2, box=1.0, clustered=False, p=8),
        # one adaptive leapfrog step with the full periodic force on a 96^3 box
        dict(name="step_96c", op="step", N=96 ** 3, K=24, R=2, box=1.0, clustered=True, p=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["forces", "forces", "train", "adjoint", "density", "batch", "bin", "far", "total", "step"])
    if op == "batch":
        lo = _log_int(rng, 3000, 12000)
        return dict(op=op, boxes=rng.randint(3, 48), n_lo=lo, n_hi=_log_int(rng, 4 * lo, 500000),
                    sizes=rng.randrange(1 << 20), clustered=rng.random() < 0.7)
    top = {"forces": 30e6, "train": 4e6, "adjoint": 12e6, "density": 10e6, "bin": 60e6, "far": 6e6, "total": 4e6,
           "step": 3e6}[op]
    N = _log_int(rng, 3000, top)
    c = dict(op=op, N=N, K=0, box=rng.choice([1.0, 1.0, 3.7, 250.0]))
    if op == "bin":
        c.update(K=rng.choice([0, 0, 7, 32, 64, 101, 128]), clustered=rng.random() < 0.5)
    else:
        c.update(R=2 if op in ("far", "total", "step") else rng.choice([2, 2, 2, 2, 1, 3]),
                 clustered=rng.random() < 0.6)
    # 40 to 90 particles per cell; at least the stencil of R = 3
    c["K"] = c["K"] or max(7, int(round((N / rng.uniform(40, 90)) ** (1 / 3))))
    if op == "density":
        c["b"] = rng.choice([0.1, 0.2, 0.2, 1.5])
    if op in ("far", "total", "step"):
        c.update(K=min(c["K"], 48), p=rng.choice([4, 6, 8, 8]))
    return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _gen(seed, salt=0):
    return torch.Generator(device=DEV).manual_seed((int(seed) * 1000003 + salt) % (1 << 62))


def _positions(N, K, box, clustered, seed, salt=0):
    """FP32 [N, 3] in [0, box): uniform, or the clustered recipe."""
    g = _gen(seed, salt)
    if not clustered or N < 200:
        x = torch.rand((N, 3), generator=g, device=DEV)
    else:
        n_cl = N - int(round(0.4 * N))
        n_sph = max(1, min(N // 512, n_cl // 20))
        mass = 20.0 * (1.0 - torch.rand(n_sph, generator=g, device=DEV, dtype=F64)) ** (-1.0 / 0.9)
        raw = (mass - 20.0) * ((n_cl - 20 * n_sph) / (mass - 20.0).sum())
        counts = 20 + raw.floor().long()
        left = n_cl - int(counts.sum())
        counts[(raw - raw.floor()).argsort(descending=True, stable=True)[:left]] += 1
        scale = 0.3 / K * (counts.double() / 64.0) ** (1.0 / 3.0)
        centre = torch.rand((n_sph, 3), generator=g, device=DEV, dtype=F64)
        of = torch.repeat_interleave(torch.arange(n_sph, device=DEV), counts)
        u = torch.rand(n_cl, generator=g, device=DEV, dtype=F64).clamp_(1e-12, 1 - 1e-12)
        v = torch.randn((n_cl, 3), generator=g, device=DEV)
        v /= v.norm(dim=1, keepdim=True)
        x = torch.empty((N, 3), device=DEV)
        x[:n_cl] = (centre[of] + (scale[of] / (u ** (-2.0 / 3.0) - 1.0).sqrt())[:, None] * v).remainder_(1.0).float()
        del of, u, v
        x[n_cl:] = torch.rand((N - n_cl, 3), generator=g, device=DEV)
        x = x[torch.randperm(N, generator=g, device=DEV)]
    if box != 1.0:
        x *= box
    x[x >= box] = 0.0
    return x


def _eps(N, box):
    return box / (40.0 * N ** (1.0 / 3.0))


def _top_hat(c):
    """The density radius: b mean spacings, inside the near field."""
    return min(c["b"] * c["box"] / c["N"] ** (1.0 / 3.0), c["R"] * c["box"] / c["K"])


def _sizes(c):
    rng = random.Random(c["sizes"])
    out = []
    for _ in range(c["boxes"]):
        N = _log_int(rng, c["n_lo"], c["n_hi"])
        out.append(dict(N=N, K=max(5, int(round((N / 64.0) ** (1 / 3)))), R=2, eps=_eps(N, 1.0), box=1.0))
    return out


def _inputs(c, seed):
    """Every array of the call, made from the seed alone."""
    if c["op"] == "batch":
        return dict(pos=torch.cat([_positions(b["N"], b["K"], 1.0, c["clustered"], seed, q + 1)
                                   for q, b in enumerate(_sizes(c))]))
    N, box = c["N"], c["box"]
    d = dict(pos=_positions(N, c["K"], box, c["clustered"], seed))
    g = _gen(seed, 77)
    if c["op"] in ("train", "adjoint"):
        d["g"] = torch.randn((N, 3), generator=g, device=DEV)
    if c["op"] == "step":
        # accelerations of the size a clustered box has; velocities that move a particle by a
        # small part of the softening in one step
        v = 0.05 / math.sqrt(box)
        d["vel"] = v * torch.randn((N, 3), generator=g, device=DEV)
        d["acc"] = 2.0 / box ** 2 * torch.randn((N, 3), generator=g, device=DEV)
        d["dt"] = torch.full((1,), 0.02 * _eps(N, box) / v, dtype=F64, device=DEV)
    return d


ETA = 0.2  # of the step criterion


def prepare(case, seed):
    c = dict(case)
    s = _inputs(c, seed)
    s["case"] = c
    if c["op"] == "batch":
        s["batch"] = nf.BatchedNearField(_sizes(c), device=DEV)
        s["batch"].pos.copy_(s["pos"])
        s["batch"].capture()
        return s
    if c["op"] == "train":
        s["pos"].requires_grad_(True)
    if c["op"] in ("far", "total", "step"):
        s["far"] = nf.FarField(c["K"], c["R"], c["p"], c["box"], device=DEV)
    if c["op"] == "step":
        N, K, R = c["N"], c["K"], c["R"]
        s["ws"] = torch.empty(_lib.nf_workspace_bytes(N, K, R), dtype=torch.uint8, device=DEV)
        s["ws_far"] = torch.empty(_lib.nf_far_workspace_bytes(N, K, c["p"]), dtype=torch.uint8, device=DEV)
        s["prm"] = _lib.make_step_params(ETA)
    return s


def run(state):
    s, c = state, state["case"]
    op = c["op"]
    if op == "batch":
        return s["batch"](s["pos"])
    if op == "bin":
        off, rel, perm = nf.bin_particles(s["pos"], c["box"], c["K"])
        # the .w of a row holds the bits of its index: returned as the whole number that it is
        return off, rel[:, :3], rel.view(torch.int32)[:, 3], perm
    if op == "far":
        return s["far"](s["pos"])
    eps = _eps(c["N"], c["box"])
    if op == "forces":
        return nf.forces(s["pos"], c["box"], c["K"], c["R"], eps)
    if op == "adjoint":
        return nf.forces_adjoint(s["pos"], s["g"], c["box"], c["K"], c["R"], eps)
    if op == "density":
        return nf.forces_density(s["pos"], c["box"], c["K"], c["R"], eps, _top_hat(c))
    if op == "train":
        acc = nf.near_field(s["pos"], c["box"], c["K"], c["R"], eps)
        grad, = torch.autograd.grad(acc, s["pos"], s["g"])
        return acc.detach(), grad
    if op == "total":
        return s["far"].total(s["pos"], eps)
    f = s["far"]
    _lib.nf_kdk_step_far(s["pos"], s["vel"], s["acc"], c["box"], c["K"], c["R"], eps, c["p"], f.derivs, s["dt"],
                         s["prm"], s["ws"], s["ws_far"])
    return s["pos"], s["vel"], s["acc"], s["dt"]


# ---------------------------------------------------------------------------
# What a call cannot do without
# ---------------------------------------------------------------------------

def _pairs(N, K, R, clustered):
    """Ordered pairs of the (2R+1)^3 stencil (expected, by the recipe)."""
    return N * float(N) * (2 * R + 1) ** 3 / K ** 3 * (CLUSTERED_PAIRS if clustered else 1.0)


# Flops of one unordered pair applied to both particles: separation 3, r^2 5, r^-3 3, two
# accumulations of f d 12; the density adds b^2 - r^2 and two sums; the adjoint 3 differences of g,
# d.v 5, the scale of d 2, J v 6 + 3, two sums 6 on top of separation, r^2 and r^-3.
PAIR_FLOPS = {"forces": 23.0, "density": 27.0, "adjoint": 42.0}


def work(case):
    c = dict(case)
    op = c["op"]
    if op == "batch":
        b = _sizes(c)
        return {"bytes": 24.0 * sum(x["N"] for x in b),
                "flops": 0.5 * PAIR_FLOPS["forces"] * sum(_pairs(x["N"], x["K"], 2, c["clustered"]) for x in b)}
    N, K = float(c["N"]), float(c["K"])
    if op == "bin":
        return {"bytes": 32.0 * N + 4.0 * K ** 3, "flops": 9.0 * N}
    near = 0.5 * _pairs(c["N"], c["K"], c["R"], c["clustered"])
    fwd, adj = near * PAIR_FLOPS["forces"], near * PAIR_FLOPS["adjoint"]
    far = 0.0
    tensor = 0.0
    if op in ("far", "total", "step"):
        p = c["p"]
        nt, nr, half = (p + 3) * (p + 2) * (p + 1) / 6, (p + 1) ** 2, K * K * (K / 2 + 1)
        # multipoles and the Taylor gradient per particle, two 3-D transforms of (p+1)^2 real fields, the product
        far = N * (2 * nt + 6 * nt) + 2 * nr * 2.5 * K ** 3 * math.log2(K ** 3) + half * nr * nr / 6 * 4
        tensor = 8.0 * nr * half  # the transformed derivatives, read once
    return {
        "forces": {"bytes": 24 * N, "flops": fwd},
        "train": {"bytes": 48 * N, "flops": fwd + adj},
        "adjoint": {"bytes": 36 * N, "flops": adj},
        "density": {"bytes": 28 * N, "flops": near * PAIR_FLOPS["density"]},
        "far": {"bytes": 36 * N + tensor, "flops": far},
        "total": {"bytes": 24 * N + tensor, "flops": fwd + far},
        "step": {"bytes": 72 * N + tensor, "flops": fwd + far + 18 * N},
    }[op]


# ---------------------------------------------------------------------------
# The same outputs in 64 bits
# ---------------------------------------------------------------------------

class _Cells:
    """Particles grouped by cell: the cell rule is t = x (K / box), c = floor(t) mod K in FP64."""

    def __init__(self, pos, box, K):
        t = pos.double() * (K / box)
        c = t.floor()
        self.K, self.w, self.rel = K, box / K, (t - c) - 0.5
        c = c.long() % K
        self.cell = (c[:, 0] * K + c[:, 1]) * K + c[:, 2]
        self.order = torch.argsort(self.cell, stable=True)
        self.count = torch.bincount(self.cell, minlength=K ** 3)
        self.start = torch.cumsum(self.count, 0) - self.count


def _near(pos, box, K, R, eps, g=None, b=None, pairs_at_once=1 << 25):
    """FP64 near-field sums over the (2R+1)^3 cells: accelerations, the adjoint for g, or (a, rho) for b."""
    N = pos.shape[0]
    cl = _Cells(pos, box, K)
    x = cl.rel[cl.order]          # cell-centred, cell units
    cell = cl.cell[cl.order]
    gs = g.double()[cl.order] if g is not None else None
    es = 2.16 * eps / cl.w
    out = torch.zeros((N, 3), dtype=F64, device=pos.device)
    rho = torch.zeros(N, dtype=F64, device=pos.device)
    i, j, k = cell // (K * K), cell // K % K, cell % K
    for a in range(-R, R + 1):
        for e in range(-R, R + 1):
            for d in range(-R, R + 1):
                other = ((i + a) % K * K + (j + e) % K) * K + (k + d) % K
                n, first = cl.count[other], cl.start[other]
                ends = torch.cumsum(n, 0)
                shift = torch.tensor([a, e, d], dtype=F64, device=pos.device)
                lo = 0
                while lo < N:
                    base = int(ends[lo - 1]) if lo else 0
                    hi = max(lo + 1, int(torch.searchsorted(ends, base + pairs_at_once, right=True)))
                    m = n[lo:hi]
                    sink = torch.repeat_interleave(torch.arange(lo, hi, device=pos.device), m)
                    if sink.numel():
                        src = first[sink] + torch.arange(sink.numel(), device=pos.device) - (ends - n)[sink] + base
                        dx = x[src] - x[sink] + shift
                        r2 = (dx * dx).sum(1)
                        r = r2.sqrt()
                        u = r / es
                        soft = u < 1
                        safe = torch.where(soft, torch.ones_like(r), r)
                        f = torch.where(soft, (10 - 15 * u + 6 * u * u) / es ** 3, safe ** -3)
                        if g is None:
                            v = f[:, None] * dx
                        else:
                            dg = gs[src] - gs[sink]
                            near = torch.where(r > 0, -15 / (es ** 4 * r.clamp_min(1e-300)) + 12 / es ** 5, 0 * r)
                            h = torch.where(soft, near, -3 * safe ** -5)
                            v = f[:, None] * dg + (h * (dx * dg).sum(1))[:, None] * dx
                        out[lo:hi] += torch.segment_reduce(v, "sum", lengths=m, unsafe=True)
                        if b is not None:
                            t = (1 - r2 * (cl.w / b) ** 2).clamp_min(0)
                            rho[lo:hi] += torch.segment_reduce(t, "sum", lengths=m, unsafe=True)
                    lo = hi
    res = torch.empty_like(out)
    res[cl.order] = out / (N * cl.w ** (2 if g is None else 3))
    if b is None:
        return res
    dens = torch.empty_like(rho)
    dens[cl.order] = rho
    return res, dens


def _terms(p):
    return [(a, b, c) for a in range(p + 1) for b in range(p + 1 - a) for c in range(p + 1 - a - b)]


def _cartesian(g, X, Y, Z, p):
    """All derivatives up to order p of a radial function from g[m] = (r^-1 d/dr)^m (Hermite recursion)."""
    layers = {(0, 0, 0): list(g)}
    for n in range(1, p + 1):
        for t, u, v in [q for q in _terms(n) if sum(q) == n]:
            ax, X1 = (0, X) if t else (1, Y) if u else (2, Z)
            one, two = [t, u, v], [t, u, v]
            one[ax] -= 1
            two[ax] -= 2
            low = layers[tuple(one)]
            lower = layers[tuple(two)] if two[ax] >= 0 else None
            layers[t, u, v] = [X1 * low[m + 1] + (one[ax] * lower[m + 1] if lower else 0) for m in range(p + 1 - n)]
    return torch.stack([layers[q][0] for q in _terms(p)])


def _derivatives(K, R, p, dev):
    """[terms, K, K, K]: derivatives of the periodic potential of a unit box (uniform background
    included) at every cell offset, without the one image that the near field holds."""
    alpha, hmax = 4.5, 13
    c = torch.arange(K, device=dev)
    c = torch.where(c > K // 2, c - K, c).double()
    gx, gy, gz = [q.reshape(-1) / K for q in torch.meshgrid(c, c, c, indexing="ij")]
    near = torch.maximum(torch.maximum(gx.abs(), gy.abs()), gz.abs()) < (R + 0.5) / K
    D = torch.zeros((len(_terms(p)), K ** 3), dtype=F64, device=dev)
    for n in [(a, b, e) for a in (-1, 0, 1) for b in (-1, 0, 1) for e in (-1, 0, 1)]:
        X, Y, Z = gx + n[0], gy + n[1], gz + n[2]
        r2 = X * X + Y * Y + Z * Z
        r = r2.sqrt()
        safe = torch.where(r > 0, r, torch.ones_like(r))
        gauss = torch.exp(-alpha ** 2 * r2) / (alpha * math.sqrt(math.pi))
        B, coul = [torch.erfc(alpha * safe) / safe], [1 / safe]
        for m in range(1, p + 1):
            B.append(((2 * m - 1) * B[-1] + (2 * alpha ** 2) ** m * gauss) / safe ** 2)
            coul.append((2 * m - 1) * coul[-1] / safe ** 2)
        erfc = [(-1) ** m * B[m] for m in range(p + 1)]
        if n == (0, 0, 0):
            y = (alpha * r) ** 2
            g = []
            for m in range(p + 1):
                s, term = torch.zeros_like(r), torch.ones_like(r)
                for q in range(80):
                    s = s + term / (2 * (q + m) + 1)
                    term = -term * y / (q + 1)
                series = 2 * alpha / math.sqrt(math.pi) * (-2 * alpha ** 2) ** m * s
                erf = torch.where(y < 4, series, (-1) ** m * (coul[m] - B[m]))
                g.append(torch.where(near, -erf, erfc[m]))
        else:
            g = erfc
        D += _cartesian(g, X, Y, Z, p)
    h = torch.arange(-hmax, hmax + 1, device=dev).double()
    kx, ky, kz = [2 * math.pi * q.reshape(-1) for q in torch.meshgrid(h, h, h, indexing="ij")]
    k2 = kx * kx + ky * ky + kz * kz
    keep = (k2 > 0) & (k2 <= (2 * math.pi * hmax) ** 2)
    kx, ky, kz, k2 = kx[keep], ky[keep], kz[keep], k2[keep]
    weight = 4 * math.pi * torch.exp(-k2 / (4 * alpha ** 2)) / k2
    for lo in range(0, K ** 3, 4096):
        s = slice(lo, lo + 4096)
        phase = gx[s, None] * kx + gy[s, None] * ky + gz[s, None] * kz
        cos, sin = phase.cos(), phase.sin()
        # the n-th derivative of cos is cos, -sin, -cos, sin
        for q, (a, b, e) in enumerate(_terms(p)):
            o = a + b + e
            trig, sign = (cos, 1 if o % 4 == 0 else -1) if o % 2 == 0 else (sin, -1 if o % 4 == 1 else 1)
            D[q, s] += sign * (trig @ (weight * kx ** a * ky ** b * kz ** e))
    D[0] -= math.pi / alpha ** 2
    return D.reshape(-1, K, K, K)


def _far(pos, box, K, R, p):
    """FP64 far-field accelerations: multipoles, convolution with the derivatives, Taylor series."""
    N = pos.shape[0]
    cl = _Cells(pos, box, K)
    x = (cl.rel.float().double() / K)[cl.order]  # the stored particle state is the FP32 offset
    terms = _terms(p)
    index = {t: q for q, t in enumerate(terms)}
    px = [[x[:, d] ** e for e in range(p + 1)] for d in range(3)]
    M = torch.stack([torch.segment_reduce(px[0][a] * px[1][b] * px[2][c], "sum", lengths=cl.count, unsafe=True)
                     for a, b, c in terms])
    axes = (1, 2, 3)
    Mh = torch.fft.rfftn(M.reshape(-1, K, K, K), dim=axes)
    Dh = torch.fft.rfftn(_derivatives(K, R, p, pos.device), dim=axes)
    fact = [math.factorial(q) for q in range(p + 1)]
    T = torch.empty((len(terms), K ** 3), dtype=F64, device=pos.device)
    for q, n in enumerate(terms):
        acc = torch.zeros_like(Mh[0])
        for k in _terms(p - sum(n)):
            co = (-1.0) ** sum(k) / (fact[n[0]] * fact[n[1]] * fact[n[2]] * fact[k[0]] * fact[k[1]] * fact[k[2]])
            acc += co * Dh[index[n[0] + k[0], n[1] + k[1], n[2] + k[2]]] * Mh[index[k]]
        T[q] = torch.fft.irfftn(acc, s=(K, K, K), dim=(0, 1, 2)).reshape(-1)
    out = torch.zeros((N, 3), dtype=F64, device=pos.device)
    cell = cl.cell[cl.order]
    for q, n in enumerate(terms):
        Tq = T[q][cell]
        for d in range(3):
            if n[d]:
                e = [n[0], n[1], n[2]]
                e[d] -= 1
                out[:, d] += n[d] * Tq * px[0][e[0]] * px[1][e[1]] * px[2][e[2]]
    res = torch.empty_like(out)
    res[cl.order] = out / (N * box ** 2)  # unit-box potential of unit masses -> box units, m = 1/N
    return res


def exact(case, seed):
    c = dict(case)
    op = c["op"]
    if op == "bin":
        cells = _Cells(_inputs(c, seed)["pos"], c["box"], c["K"])
        return None, cells.rel[cells.order], None, None
    if op == "batch":
        boxes = _sizes(c)
        if sum(_pairs(b["N"], b["K"], 2, c["clustered"]) for b in boxes) > EXACT_PAIRS:
            return None
        parts = _inputs(c, seed)["pos"].split([b["N"] for b in boxes])
        return torch.cat([_near(x, 1.0, b["K"], 2, b["eps"]) for x, b in zip(parts, boxes)])
    N, K, R, box = c["N"], c["K"], c["R"], c["box"]
    if op != "far" and _pairs(N, K, R, c["clustered"]) * (3 if op in ("train", "adjoint") else 1) > EXACT_PAIRS:
        return None
    if op in ("far", "total", "step") and K > 40:
        return None
    d = _inputs(c, seed)
    pos, eps = d["pos"], _eps(N, box)
    if op == "far":
        return _far(pos, box, K, R, c["p"])
    if op == "forces":
        return _near(pos, box, K, R, eps)
    if op == "adjoint":
        return _near(pos, box, K, R, eps, g=d["g"])
    if op == "density":
        return _near(pos, box, K, R, eps, b=_top_hat(c))
    if op == "train":
        return _near(pos, box, K, R, eps), _near(pos, box, K, R, eps, g=d["g"])
    if op == "total":
        return _near(pos, box, K, R, eps) + _far(pos, box, K, R, c["p"])
    dt = float(d["dt"])
    vel = d["vel"].double() + 0.5 * dt * d["acc"].double()
    x = ((pos.double() + dt * vel.float().double()) % box).float()  # the state is FP32
    x[x >= box] = 0.0
    acc = _near(x, box, K, R, eps) + _far(x, box, K, R, c["p"])
    vel = vel + 0.5 * dt * acc
    cl = _Cells(x, box, K)
    v2, a2 = (vel * vel).sum(1), (acc * acc).sum(1)
    peak = torch.zeros(K ** 3, dtype=F64, device=x.device).scatter_reduce_(0, cl.cell, a2, "amax")
    mean = torch.zeros(K ** 3, dtype=F64, device=x.device).index_add_(0, cl.cell, v2) / cl.count.clamp_min(1)
    ratio = (mean / peak.clamp_min(1e-300)).sqrt()[peak > 0].min()
    return x.double(), vel, acc, (ETA * torch.maximum(ratio, (v2.mean() / a2.max()).sqrt())).reshape(1)
