"""What the speed of this library is judged by: the calls a user's program makes.

A user builds a grid and a plan once, then for every noise map runs the
kernel table, the block sampling and the factorisation (a "step"), applies
the factored blocks to vectors inside a solver, convolves maps with the beam
kernels, and samples the blocks between rings or the tile-coupled band blocks
of a DP grid.  Inputs follow the workloads of this repository: Gaussian
beams, the l^4 prior, lognormal inverse noise with a masked band around the
equator (white maps for the vectors that are applied to or convolved).

`exact` computes the same outputs in 64 bits from the formulas, with torch
and numpy only: ring geometry, Legendre sums per separation, explicit sums
over pixel arcs, and an unblocked Cholesky.
"""
import math

import numpy as np
import torch

from paper_1504_04653_gb300 import sympix as S

ARCMIN = math.pi / (180.0 * 60.0)


# -- the cases ------------------------------------------------------------------

def listed():
    return [
        # the smallest grid: a whole step in FP64, where launches and latency count
        dict(name="step_64", kind="step", lmax=64, fwhm=180.0, fwhm_hi=180.0, nops=1, band=20.0,
             sample="fp64", factor="fp64", graph=False),
        # an ordinary grid in FP64, the entry points' default arithmetic
        dict(name="step_500_fp64", kind="step", lmax=500, fwhm=30.0, fwhm_hi=30.0, nops=1, band=20.0,
             sample="fp64", factor="fp64", graph=False),
        # several operators (beams and noise maps) near FP64 accuracy on the FP32 pipes
        dict(name="step_750_fp32x2", kind="step", lmax=750, fwhm=16.0, fwhm_hi=20.0, nops=3, band=10.0,
             sample="fp32x2", factor="fp32x2", graph=False),
        # FP32 contraction with an FP64 factor, replayed from captured graphs
        dict(name="step_1500_mixed", kind="step", lmax=1500, fwhm=10.0, fwhm_hi=10.0, nops=1, band=20.0,
             sample="fp32", factor="fp64", graph=True),
        # the paper's resolution, FP32 contraction and factor, replayed from captured graphs
        dict(name="step_3000_fp32", kind="step", lmax=3000, fwhm=5.0, fwhm_hi=5.0, nops=1, band=20.0,
             sample="fp32", factor="fp32", graph=True),
        # wide beams: many coupled rings and long arcs (table and sampling)
        dict(name="sample_1000_wide", kind="sample", lmax=1000, fwhm=10.0, fwhm_hi=60.0, nops=4, band=15.0,
             sample="fp32", factor="", graph=False),
        # one preconditioner application in a solver's iteration, two sizes
        dict(name="apply_500", kind="apply", lmax=500, fwhm=30.0, fwhm_hi=30.0, nops=2, band=20.0,
             sample="fp64", factor="fp64", graph=False),
        dict(name="apply_3000", kind="apply", lmax=3000, fwhm=5.0, fwhm_hi=5.0, nops=1, band=20.0,
             sample="fp64", factor="fp64", graph=False),
        # beam convolution of maps: the paper's resolution, and a few wide beams
        dict(name="convolve_3000", kind="convolve", lmax=3000, fwhm=5.0, fwhm_hi=5.0, nops=1, band=0.0,
             sample="fp64", factor="", graph=False),
        dict(name="convolve_400_wide", kind="convolve", lmax=400, fwhm=40.0, fwhm_hi=120.0, nops=3, band=0.0,
             sample="fp64", factor="", graph=False),
        # the blocks between neighbouring rings (line or multi-ring preconditioners)
        dict(name="coupling_1500", kind="coupling", lmax=1500, fwhm=10.0, fwhm_hi=10.0, nops=1, band=20.0,
             sample="fp64", factor="", graph=False),
        # the paper's own DP grid with k x k tiles: dense band blocks
        dict(name="tiles_255_k4", kind="tiles", lmax=255, k=4, fwhm=60.0, fwhm_hi=60.0, nops=1, band=20.0,
             sample="fp64", factor="", graph=False),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "sample", "apply", "apply", "convolve", "convolve", "coupling",
                       "tiles"])
    c = dict(kind=kind, band=round(rng.uniform(0.0, 30.0), 1), factor="", graph=False)
    if kind in ("step", "apply"):
        # beams matched to the band limit, as in every workload with a factor, and masks
        # up to its 20 degrees: every block is then positive definite
        c["band"] = round(rng.uniform(0.0, 20.0), 1)
        c["lmax"] = _logint(rng, 64, 3000 if kind == "step" else 2500)
        most = 1 if c["lmax"] > 1000 else 4
        c["nops"] = rng.randint(1, most)
        c["fwhm"] = round(rng.uniform(11520.0, 15000.0) / c["lmax"], 2)
        c["fwhm_hi"] = round(min(c["fwhm"] * rng.uniform(1.0, 1.25), 15000.0 / c["lmax"]), 2)
        c["sample"], c["factor"] = rng.choice([("fp64", "fp64"), ("fp64", "fp64"), ("fp32", "fp64"), ("fp32", "fp32"),
                                               ("fp32x2", "fp32x2")])
        if kind == "step":
            c["graph"] = rng.random() < 0.5
    elif kind == "sample":
        c["lmax"] = _logint(rng, 150, 1000)
        c["nops"] = rng.randint(1, 4)
        c["fwhm"] = round(rng.uniform(10000.0, 25000.0) / c["lmax"], 2)
        c["fwhm_hi"] = round(c["fwhm"] + rng.uniform(0.0, 35000.0) / c["lmax"], 2)
        c["sample"] = rng.choice(["fp32", "fp32", "fp32x2", "fp64"]) if c["lmax"] < 400 else rng.choice(["fp32", "fp32x2"])
    elif kind == "convolve":
        c["lmax"] = _logint(rng, 64, 3000)
        c["nops"] = rng.randint(1, 1 if c["lmax"] > 1000 else 4)
        c["fwhm"] = round(rng.uniform(10000.0, 20000.0) / c["lmax"], 2)
        c["fwhm_hi"] = round(c["fwhm"] * (rng.uniform(1.0, 3.0) if c["lmax"] <= 1000 else 1.0), 2)
        c["sample"] = rng.choice(["fp64", "fp64", "fp32", "fp32x2"])
    elif kind == "coupling":
        c["lmax"] = _logint(rng, 64, 1500)
        c["nops"] = rng.randint(1, 1 if c["lmax"] > 500 else 3)
        c["fwhm"] = c["fwhm_hi"] = round(rng.uniform(10000.0, 15000.0) / c["lmax"], 2)
        c["sample"] = "fp64"
    else:
        c["k"] = rng.choice([2, 3, 4, 5])
        c["lmax"] = _logint(rng, 63, 255)
        c["nops"] = 1
        c["fwhm"] = c["fwhm_hi"] = round(15000.0 / c["lmax"], 2)
        c["sample"] = rng.choice(["fp64", "fp32", "fp32x2"])
    return c


def _fwhms(case):
    """FWHM of every operator in arcminutes, evenly from fwhm to fwhm_hi."""
    n = case["nops"]
    return [case["fwhm"] + (case["fwhm_hi"] - case["fwhm"]) * (i / (n - 1) if n > 1 else 0.0) for i in range(n)]


def _sigma(fwhm):
    return fwhm * ARCMIN / math.sqrt(8.0 * math.log(2.0))


def _radii(case):
    """Support radius of every operator: where the Gaussian envelope falls to 1e-10."""
    return np.array([_sigma(f) * math.sqrt(2.0 * math.log(1e10)) for f in _fwhms(case)])


def _spectra(case):
    """b_l and d_l of every operator."""
    ell = np.arange(case["lmax"] + 1, dtype=np.float64)
    bl = np.stack([np.exp(-0.5 * ell * (ell + 1.0) * _sigma(f) ** 2) for f in _fwhms(case)])
    top = case["lmax"] * (case["lmax"] + 1.0)
    dl = np.stack([(ell * (ell + 1.0) / top) ** 2] * case["nops"])
    return bl, dl


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _maps(case, seed, theta, nring, offset, stride, npix):
    """Seeded inverse-noise maps and white maps [nops, npix]."""
    dev = _device()
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    z = torch.randn(2, case["nops"], npix, generator=gen, dtype=torch.float64, device=dev)
    masked = np.zeros(npix, dtype=bool)
    for j in np.nonzero(np.abs(0.5 * math.pi - theta) < case["band"] * math.pi / 180.0)[0]:
        masked[int(offset[j]) + int(stride[j]) * np.arange(int(nring[j]))] = True
    ninv = torch.exp(0.3 * z[0])
    ninv[:, torch.from_numpy(masked).to(dev)] = 0.0
    return ninv, z[1].contiguous()


# -- preparing and running --------------------------------------------------------

class State:
    """What a user's program holds before the call."""


def prepare(case, seed):
    s = State()
    s.case = case
    kind, nops = case["kind"], case["nops"]
    if kind == "tiles":
        s.grid = S.Grid(case["lmax"], k=case["k"], layout="dp")
    else:
        s.grid = S.Grid(case["lmax"])
    g = s.grid
    s.plan = S.Plan(g, _radii(case))
    bl, dl = _spectra(case)
    s.bl, s.dl = torch.from_numpy(bl).cuda(), torch.from_numpy(dl).cuda()
    s.ninv, s.x = _maps(case, seed, g.theta, g.nring, g.ring_offset, g.ring_stride, int(g.npix))
    if kind in ("step", "sample", "tiles", "apply"):
        nbytes, _ = s.plan.blocks_size("pband")
        s.blocks = torch.zeros(nbytes // 8, dtype=torch.float64, device="cuda")
    if kind in ("step", "apply"):
        s.info = torch.zeros(s.plan.nblocks, dtype=torch.int32, device="cuda")
    if kind == "step" and case["graph"]:
        s.step = S.Step(s.plan, s.bl, s.dl, s.ninv, s.blocks, s.info, sample_precision=case["sample"],
                        factor_precision=case["factor"])
    if kind == "coupling":
        nbytes, _ = s.plan.coupling_size(1)
        s.out = torch.zeros(nbytes // 8, dtype=torch.float64, device="cuda")
    if kind in ("apply", "convolve", "coupling"):
        S.sympix_kernel_table(s.plan, s.bl, s.dl)
    if kind == "apply":
        S.sympix_sample_blocks(s.plan, s.ninv, precision=case["sample"], out=s.blocks)
        S.sympix_factor_blocks(s.plan, s.blocks, precision=case["factor"], info=s.info)
    if kind in ("apply", "convolve"):
        s.y = torch.zeros_like(s.x)
    return s


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "step":
        if case["graph"]:
            s.step.launch()
        else:
            S.sympix_kernel_table(s.plan, s.bl, s.dl)
            S.sympix_sample_blocks(s.plan, s.ninv, precision=case["sample"], out=s.blocks)
            S.sympix_factor_blocks(s.plan, s.blocks, precision=case["factor"], info=s.info)
        return {"blocks": s.blocks, "info": s.info}
    if kind in ("sample", "tiles"):
        S.sympix_kernel_table(s.plan, s.bl, s.dl)
        return {"blocks": S.sympix_sample_blocks(s.plan, s.ninv, precision=case["sample"], out=s.blocks)}
    if kind == "apply":
        return {"y": S.sympix_apply(s.plan, s.blocks, s.info, s.x, out=s.y)}
    if kind == "convolve":
        return {"g": S.sympix_convolve(s.plan, s.x, precision=case["sample"], out=s.y)}
    return {"blocks": S.sympix_sample_coupling(s.plan, s.ninv, delta=1, out=s.out)}


# -- the geometry, in numpy ---------------------------------------------------------

def _gl_theta(N):
    """Roots of P_N(cos theta), north to south, by Newton's method."""
    j = np.arange(N // 2)
    t = math.pi * (j + 0.75) / (N + 0.5)
    for _ in range(6):
        u = 2.0 * np.sin(0.5 * t) ** 2
        p, d = 1.0 - u, -u  # P_1 and P_1 - P_0
        for l in range(1, N):
            d = (l * d - (2 * l + 1) * u * p) / (l + 1)
            p = p + d
        c, s = np.cos(t), np.sin(t)
        t = t + p * s / (N * ((p - d) - c * p))
    return np.concatenate([t, [0.5 * math.pi] if N % 2 else [], math.pi - t[::-1]])


def _smooth(v):
    for f in (2, 3, 5):
        while v % f == 0:
            v //= f
    return v == 1


def _next_smooth(v):
    while not _smooth(v):
        v += 1
    return v


def _greedy_counts(lmax, theta):
    """Per-ring counts from the equator outward, target 2 (lmax + 1) sin theta, at least 8."""
    N = lmax + 1
    e = (N - 1) // 2 if N % 2 else N // 2 - 1
    n = np.zeros(N, np.int64)
    n[e] = _next_smooth(max(8, math.ceil(2.0 * N * math.sin(theta[e]))))
    for j in range(e - 1, -1, -1):
        t, prev = 2.0 * N * math.sin(theta[j]), int(n[j + 1])
        fit = [prev] + [prev * b // a for a, b in ((6, 5), (5, 4), (4, 3), (2, 1), (3, 1)) if prev * b % a == 0]
        n[j] = min(c for c in fit if c == prev or (c >= 8 and c >= t))
    n[N - 1 - np.arange(e + 1)] = n[:e + 1]
    return n


def _dp_counts(lmax, k, theta):
    """Tiles per band by dynamic programming (least squared excess over the
    polar bound; neighbouring ratios 1, 2, 3, 4/3, 5/4, 6/5, two equal bands
    before a change), mirrored; returns pixels per ring."""
    N, nb = len(theta), len(theta) // (2 * k)
    thr = max(100.0, lmax / 100.0)
    m = np.arange(lmax + 1.0)
    alpha = []
    for i in range(nb):
        th = theta[i * k + k - 1]
        a = m * m - 2.0 * m * math.cos(th)
        ok = (a >= 0.0) & (np.sqrt(np.maximum(a, 0.0)) - lmax * math.sin(th) > thr)
        mm = int(np.argmax(ok)) if ok.any() else lmax + 1
        alpha.append((2 * mm + 1 + k - 1) // k)
    t0 = _next_smooth(alpha[0])
    layer = [{t0: ((t0 - alpha[0]) ** 2, t0)}]
    for i in range(1, nb):
        a, new = alpha[i], {}
        for tp, (cost, before) in layer[-1].items():
            for x, y in ((3, 1), (2, 1), (1, 1), (4, 3), (5, 4), (6, 5)):
                if tp * x % y:
                    continue
                t = tp * x // y
                if a <= t <= 3 * a and (before == tp or x == y):
                    key = (cost + (a - t) ** 2, tp)
                    if t not in new or key < new[t]:
                        new[t] = key
        layer.append(new)
    t = min(layer[-1], key=lambda v: (layer[-1][v][0], v))
    T = [t]
    for i in range(nb - 1, 0, -1):
        t = layer[i][t][1]
        T.append(t)
    T = T[::-1]
    n = np.array([k * T[min(j, N - 1 - j) // k] for j in range(N)], np.int64)
    return n


class _Sphere:
    """Rings, pixel numbering and coupled separations of a case."""

    def __init__(self, case):
        lmax, k = case["lmax"], case.get("k", 1)
        N = lmax + 1
        if case["kind"] == "tiles" and N % (2 * k):
            N += 2 * k - N % (2 * k)
        self.N, self.k, self.lmax = N, k, lmax
        self.theta = _gl_theta(N)
        self.n = _dp_counts(lmax, k, self.theta) if case["kind"] == "tiles" else _greedy_counts(lmax, self.theta)
        self.offset, self.stride = np.zeros(N, np.int64), np.full(N, k, np.int64)
        pos = 0
        for i in range(N // (2 * k)):
            for first, step in ((i * k, 1), (N - 1 - i * k, -1)):
                for r in range(k):
                    self.offset[first + step * r] = pos + r
                pos += int(self.n[first]) * k
        if k == 1 and N % 2:
            self.offset[N // 2] = pos
            pos += int(self.n[N // 2])
        self.npix = pos

    def constants(self, j, rho):
        nj, nr = int(self.n[j]), int(self.n[rho])
        g = math.gcd(nj, nr)
        return nj // g, nr // g, g

    def pair_u(self, j, rho):
        """u(z) = base + st sin^2(pi z g / (2 n_j n_rho)) of a ring pair: (base, st)."""
        ta, tb = self.theta[j], self.theta[rho]
        return 2.0 * math.sin(0.5 * (ta - tb)) ** 2, 2.0 * math.sin(ta) * math.sin(tb)

    def mmax(self, j, rho, r_s, slack=0.0):
        """Largest coupled |z| of a ring pair (-1: none)."""
        P, Q, g = self.constants(j, rho)
        par, half = (P + Q) % 2, P * Q * g
        cap = half - (half - par) % 2
        if r_s >= math.pi:
            return cap
        base, st = self.pair_u(j, rho)
        h = (2.0 * math.sin(0.5 * r_s) ** 2 * (1.0 + slack) - base) / st
        if h < 0.0:
            return -1
        if h >= 1.0:
            return cap
        m = int(math.asin(math.sqrt(h)) * 2.0 * half / math.pi)
        m -= (m - par) % 2
        return min(cap, m)

    def neighbours(self, j, r_s):
        """(rho, m) of every ring coupled to ring j."""
        got = []
        for step in (-1, 1):
            rho = j if step < 0 else j + 1
            while 0 <= rho < self.N and abs(self.theta[rho] - self.theta[j]) <= r_s:
                m = self.mmax(j, rho, r_s)
                if m >= 0:
                    got.append((rho, m))
                rho += step
        return sorted(got)

    def blocks(self, case):
        """Every (operator, ring) block: op, ring, n, w, periodic band or dense, neighbours, offset."""
        out, off = [], 0
        for o, r_s in enumerate(_radii(case)):
            shape = []
            for j in range((self.N + 1) // 2):
                near = self.neighbours(j, r_s)
                w, wrap = 0, False
                for rho, m in near:
                    P, Q, g = self.constants(j, rho)
                    w = max(w, m // Q)
                    wrap |= m >= P * Q * g - P
                shape.append((w, wrap, near))
            for j in range(self.N):
                w, wrap, near = shape[min(j, self.N - 1 - j)]
                if j != min(j, self.N - 1 - j):
                    near = sorted((self.N - 1 - rho, m) for rho, m in near)
                n = int(self.n[j])
                dense = wrap or 2 * w + 1 >= n or w > 64
                off = (off + 3) // 4 * 4
                out.append(dict(op=o, ring=j, n=n, w=w, dense=dense, near=near, off=off))
                off += n * n if dense else n * (2 * w + 1)
        return out, off


def work(case):
    """Bytes: inputs once, outputs once.  Flops: the recurrence at every
    distinct separation, two per multiply-add of the sums over coupled pixels,
    and the factor's or the substitutions' multiply-adds."""
    sph = _Sphere(case)
    nops, lmax, kind = case["nops"], case["lmax"], case["kind"]
    npix = sph.npix
    if kind == "tiles":
        k, G = case["k"], sph.N // case["k"]
        nbytes, flops = 8.0 * npix, 0.0
        for g in range(G):
            K = k * int(sph.n[g * k])
            nbytes += 8.0 * K * K
            # about 5 tiles near each tile in latitude neighbours, 3 x 3 tiles coupled
            flops += 2.0 * K * (5 * k * k) * (6 * k * k) if 0 < g < G - 1 else 2.0 * K * K * K
        return {"bytes": nbytes, "flops": flops}
    blocks, size = sph.blocks(case)
    slots = sum(m // 2 + 1 for b in blocks for rho, m in b["near"] if rho <= b["ring"] <= sph.N - 1 - rho)
    table = 9.0 * slots * lmax
    pairs = trip = elems = fact = 0.0
    for b in blocks:
        n, w = b["n"], b["w"]
        for rho, m in b["near"]:
            P, Q, g = sph.constants(b["ring"], rho)
            arc = min(m + 1, P * int(sph.n[rho]))
            pairs += n * arc / P
            trip += sum(max(0, m - d * Q + 1) for d in range(w + 1)) * n / P if not b["dense"] else n * n * arc / P
        elems += n * n if b["dense"] else n * (2 * w + 1)
        fact += n ** 3 / 6 if b["dense"] else n * 2.0 * w * w
    maps = 8.0 * nops * npix
    if kind == "step":
        return {"bytes": maps + 8.0 * elems, "flops": table + 2.0 * trip + 2.0 * fact}
    if kind == "sample":
        return {"bytes": maps + 4.0 * elems, "flops": table + 2.0 * trip}
    if kind == "apply":
        return {"bytes": 2.0 * maps + 8.0 * elems, "flops": 4.0 * elems}
    if kind == "convolve":
        return {"bytes": 2.0 * maps, "flops": 2.0 * pairs}
    return {"bytes": maps + 8.0 * elems, "flops": 4.0 * trip}


# -- the outputs in 64 bits ---------------------------------------------------------

class _Table:
    """b and d of every operator at the separations of a set of ring pairs."""

    def __init__(self, case, sph, pairs):
        """pairs: {(j, rho): m}; pairs that a mirror or a swap maps onto each other share values."""
        dev = _device()
        self.sph, self.first = sph, {}
        most = {}
        for (j, rho), m in pairs.items():
            key = self.canon(j, rho)
            most[key] = max(most.get(key, -1), m)
        us, pos = [], 0
        for (a, b), m in most.items():
            P, Q, g = sph.constants(a, b)
            base, st = sph.pair_u(a, b)
            z = np.arange((P + Q) % 2, m + 1, 2, dtype=np.float64)
            us.append(base + st * np.sin(0.5 * math.pi * z / (P * Q * g)) ** 2)
            self.first[(a, b)] = pos
            pos += len(z)
        u = torch.from_numpy(np.concatenate(us)).to(dev)
        bl, dl = _spectra(case)
        ell = 2.0 * np.arange(case["lmax"] + 1) + 1.0
        cb = torch.from_numpy(bl * ell / (4.0 * math.pi)).to(dev)
        cd = torch.from_numpy(dl * ell / (4.0 * math.pi)).to(dev)
        p, d = torch.ones_like(u), torch.zeros_like(u)
        self.b, self.d = cb[:, :1] * p, cd[:, :1] * p
        for l in range(case["lmax"]):
            d = (l * d - (2 * l + 1) * u * p) / (l + 1)
            p = p + d
            self.b.addcmul_(cb[:, l + 1:l + 2], p)
            self.d.addcmul_(cd[:, l + 1:l + 2], p)

    def canon(self, j, rho):
        N = self.sph.N
        a, b = min(j, rho), max(j, rho)
        return (a, b) if a <= N - 1 - b else (N - 1 - b, N - 1 - a)

    def values(self, which, op, j, rho, m):
        """Values at |z| = par, par + 2, ..., m."""
        P, Q, _ = self.sph.constants(j, rho)
        at = self.first[self.canon(j, rho)]
        return which[op, at:at + (m - (P + Q) % 2) // 2 + 1]


def _ring_table(case, sph, blocks, all_pairs=()):
    pairs = {}
    for b in blocks:
        for rho, m in b["near"]:
            pairs[(b["ring"], rho)] = max(m, pairs.get((b["ring"], rho), -1))
    for key, m in all_pairs:
        pairs[key] = max(m, pairs.get(key, -1))
    return _Table(case, sph, pairs)


def _ring_map(sph, maps, op, j):
    return maps[op, int(sph.offset[j]):int(sph.offset[j]) + int(sph.stride[j]) * int(sph.n[j]):int(sph.stride[j])]


def _near(z, half):
    z = torch.remainder(z, 2 * half)
    return torch.where(z > half, z - 2 * half, z)


def _kernel_rows(sph, val, j, rho, m, columns, p):
    """Kernel of pixels `columns` of ring j against pixels p of ring rho (0 where not coupled)."""
    P, Q, g = sph.constants(j, rho)
    z = _near((2 * columns + 1) * Q - (2 * p + 1) * P, P * Q * g).abs()
    return torch.where(z <= m, val[((z - (P + Q) % 2) // 2).clamp(0, len(val) - 1)], torch.zeros((), dtype=val.dtype, device=val.device))


def _arc(sph, j, rho, m, columns):
    """Pixels of ring rho that may couple to `columns` of ring j, one row each (every pixel at most once)."""
    P, Q, _ = sph.constants(j, rho)
    lo = -torch.div(-((2 * columns + 1) * Q - m - P), 2 * P, rounding_mode="floor")
    return lo[:, None] + torch.arange(min(m // P + 1, int(sph.n[rho])), device=columns.device)


def _sampled(case, sph, blocks, size, tab, ninv):
    """The sampled blocks buffer."""
    dev = ninv.device
    out = torch.zeros(size, dtype=torch.float64, device=dev)
    for b in blocks:
        o, j, n, w = b["op"], b["ring"], b["n"], b["w"]
        q = torch.arange(n, device=dev)
        if b["dense"]:
            M = torch.zeros(n, n, dtype=torch.float64, device=dev)
            for rho, m in b["near"]:
                p = torch.arange(int(sph.n[rho]), device=dev)
                B = _kernel_rows(sph, tab.values(tab.b, o, j, rho, m), j, rho, m, q[:, None], p[None, :])
                M += (B * _ring_map(sph, ninv, o, rho)) @ B.T
                if rho == j:
                    M += _kernel_rows(sph, tab.values(tab.d, o, j, j, m), j, j, m, q[:, None], q[None, :])
            out[b["off"]:b["off"] + n * n] = M.reshape(-1)
            continue
        M = torch.zeros(n, w + 1, dtype=torch.float64, device=dev)
        back = torch.arange(w + 1, device=dev)
        for rho, m in b["near"]:
            P, Q, _ = sph.constants(j, rho)
            val = tab.values(tab.b, o, j, rho, m)
            # columns c, c + P, c + 2P, ... see the same kernel values
            first = _arc(sph, j, rho, m, q[:P])
            z = (2 * q[:P, None] + 1) * Q - (2 * first + 1) * P
            zd = (z[:, :, None] - 2 * Q * back).abs()
            T = torch.where((zd <= m) & (z[:, :, None].abs() <= m),
                            val[((zd - (P + Q) % 2) // 2).clamp(0, len(val) - 1)], 0.0)
            p = torch.remainder(first[None] + Q * torch.arange(n // P, device=dev)[:, None, None], int(sph.n[rho]))
            W = torch.where(z.abs() <= m, val[((z.abs() - (P + Q) % 2) // 2).clamp(0, len(val) - 1)], 0.0)
            wp = W[None] * _ring_map(sph, ninv, o, rho)[p]
            M += torch.einsum("tcp,cpd->tcd", wp, T).reshape(n, w + 1)
            if rho == j:
                dv = tab.values(tab.d, o, j, j, m)
                M[:, :len(dv)] += dv[:w + 1]
        out[b["off"]:b["off"] + n * (w + 1)] = M.reshape(-1)
    return out


def _groups(blocks):
    """Periodic-band blocks of one width together (at most about 2 GB of columns)."""
    by = {}
    for b in blocks:
        if not b["dense"]:
            by.setdefault(b["w"], []).append(b)
    for w, bs in by.items():
        bs = sorted(bs, key=lambda b: -b["n"])
        per = max(1, int(2e9 / (8.0 * bs[0]["n"] * (2 * w + 1))))
        for i in range(0, len(bs), per):
            yield w, bs[i:i + per]


def _band_factor(w, bs, buf):
    """Column-oriented Cholesky of periodic-band blocks: C[:, i, t] = L[i+t][i],
    X[:, b, i] = L[m+b][i] (i < m = n - w) and the corner; blocks shorter than
    the longest are padded with identity columns."""
    dev, nb = buf.device, len(bs)
    top = bs[0]["n"] - w
    C = torch.zeros(nb, top + w + 1, w + 1, dtype=torch.float64, device=dev)
    X = torch.zeros(nb, w, top + w + 1, dtype=torch.float64, device=dev)
    A22 = torch.zeros(nb, w, w, dtype=torch.float64, device=dev)
    C[:, :, 0] = 1.0
    for i, b in enumerate(bs):
        n = b["n"]
        m = n - w
        M = buf[b["off"]:b["off"] + n * (w + 1)].reshape(n, w + 1)
        for d in range(w + 1):
            C[i, :m - d, d] = M[d:m, d]
        for t in range(w):
            for d in range(w + 1):
                if t - d < 0:
                    X[i, t, m + t - d] = M[m + t, d]
                else:
                    A22[i, t, t - d] = M[m + t, d]
                if d > t:  # row t couples backwards over the start of the ring
                    X[i, w + t - d, t] = M[t, d]
    idx = torch.arange(w, device=dev)[:, None] + torch.arange(w + 1, device=dev)[None, :]
    pad = torch.zeros(nb, 2 * w + 1, dtype=torch.float64, device=dev)
    for i in range(top):
        C[:, i] *= torch.rsqrt(C[:, i, :1])
        r = 1.0 / C[:, i, 0]
        if w:
            l = C[:, i, 1:]
            X[:, :, i] *= r[:, None]
            pad[:, :w] = l
            C[:, i + 1:i + 1 + w] -= l[:, :, None] * pad[:, idx]
            X[:, :, i + 1:i + 1 + w] -= X[:, :, i, None] * l[:, None, :]
    X = X[:, :, :top].contiguous()
    L22 = torch.linalg.cholesky(torch.tril(A22) + torch.tril(A22, -1).transpose(1, 2) - X @ X.transpose(1, 2)) if w else A22
    return C[:, :top], X, L22


def _factored(blocks, buf):
    """The factored blocks buffer: L where it is defined, the sampled values elsewhere."""
    out = buf.clone()
    for b in blocks:
        if b["dense"]:
            n = b["n"]
            M = buf[b["off"]:b["off"] + n * n].reshape(n, n)
            L = torch.linalg.cholesky(M)
            out[b["off"]:b["off"] + n * n] = (L + torch.triu(M, 1)).reshape(-1)
    for w, bs in _groups(blocks):
        C, X, L22 = _band_factor(w, bs, buf)
        for i, b in enumerate(bs):
            n = b["n"]
            m = n - w
            band = out[b["off"]:b["off"] + n * (w + 1)].view(n, w + 1)
            for d in range(w + 1):
                band[d:m, d] = C[i, :m - d, d]
            bord = out[b["off"] + n * (w + 1):b["off"] + n * (2 * w + 1)].view(w, n)
            bord[:, :m] = X[i, :, :m]
            bord[:, m:] = torch.tril(L22[i])
    return out


def _applied(sph, blocks, buf, x):
    """y = M^-1 x block by block."""
    y = torch.zeros_like(x)
    for b in blocks:
        if b["dense"]:
            n = b["n"]
            M = buf[b["off"]:b["off"] + n * n].reshape(n, n)
            v = _ring_map(sph, x, b["op"], b["ring"])
            _ring_map(sph, y, b["op"], b["ring"])[:] = torch.cholesky_solve(v[:, None], torch.linalg.cholesky(M))[:, 0]
    for w, bs in _groups(blocks):
        C, X, L22 = _band_factor(w, bs, buf)
        nb, top = C.shape[:2]
        v = torch.zeros(nb, top + w, dtype=torch.float64, device=x.device)
        tail = torch.zeros(nb, w, dtype=torch.float64, device=x.device)
        for i, b in enumerate(bs):
            r = _ring_map(sph, x, b["op"], b["ring"])
            v[i, :b["n"] - w], tail[i] = r[:b["n"] - w], r[b["n"] - w:]
        for i in range(top):
            v[:, i] /= C[:, i, 0]
            if w:
                v[:, i + 1:i + 1 + w] -= C[:, i, 1:] * v[:, i:i + 1]
        if w:
            v[:, top:] = 0.0
            tail = torch.cholesky_solve((tail - (X @ v[:, :top, None])[:, :, 0])[:, :, None], L22)[:, :, 0]
            v[:, :top] -= (X.transpose(1, 2) @ tail[:, :, None])[:, :, 0]
        for i in range(top - 1, -1, -1):
            s = v[:, i] - (C[:, i, 1:] * v[:, i + 1:i + 1 + w]).sum(1) if w else v[:, i]
            v[:, i] = s / C[:, i, 0]
        for i, b in enumerate(bs):
            r = _ring_map(sph, y, b["op"], b["ring"])
            r[:b["n"] - w], r[b["n"] - w:] = v[i, :b["n"] - w], tail[i]
    return y


def _convolved(sph, blocks, tab, f):
    g = torch.zeros_like(f)
    for b in blocks:
        o, j = b["op"], b["ring"]
        q = torch.arange(b["n"], device=f.device)
        acc = torch.zeros(b["n"], dtype=torch.float64, device=f.device)
        for rho, m in b["near"]:
            p = _arc(sph, j, rho, m, q)
            B = _kernel_rows(sph, tab.values(tab.b, o, j, rho, m), j, rho, m, q[:, None], p)
            acc += (B * _ring_map(sph, f, o, rho)[torch.remainder(p, int(sph.n[rho]))]).sum(1)
        _ring_map(sph, g, o, j)[:] = acc
    return g


def _coupled(case, sph, blocks, tab, ninv):
    """The blocks between rings j and j + 1."""
    outs, r_s, dev = [], _radii(case), ninv.device
    at = {(b["op"], b["ring"]): b for b in blocks}
    for o in range(case["nops"]):
        for j in range(sph.N - 1):
            k = j + 1
            P, Q, g = sph.constants(j, k)
            zmax = max(0, sph.mmax(j, k, min(2.0 * r_s[o], math.pi), 1e-9))
            K, nk = zmax // P + 1, int(sph.n[k])
            q = torch.arange(int(sph.n[j]), device=dev)
            full = K >= nk
            if full:
                r = torch.arange(nk, device=dev).expand(len(q), nk)
            else:
                lo = -torch.div(-((2 * q + 1) * Q - zmax - P), 2 * P, rounding_mode="floor")
                r = lo[:, None] + torch.arange(K, device=dev)
            M = torch.zeros(r.shape, dtype=torch.float64, device=dev)
            for rho, m in at[(o, k)]["near"]:
                if rho == j:
                    M += _kernel_rows(sph, tab.values(tab.d, o, j, k, m), j, k, m, q[:, None], r)
            far = dict(at[(o, k)]["near"])
            for rho, m in at[(o, j)]["near"]:
                if rho not in far:
                    continue
                p = _arc(sph, j, rho, m, q)
                W = _kernel_rows(sph, tab.values(tab.b, o, j, rho, m), j, rho, m, q[:, None], p)
                W = W * _ring_map(sph, ninv, o, rho)[torch.remainder(p, int(sph.n[rho]))]
                B = _kernel_rows(sph, tab.values(tab.b, o, k, rho, far[rho]), k, rho, far[rho], r[:, :, None], p[:, None, :])
                M += torch.einsum("qp,qrp->qr", W, B)
            if not full:
                M[((2 * q[:, None] + 1) * Q - (2 * r + 1) * P).abs() > zmax] = 0.0
            outs.append(M.reshape(-1))
    return torch.cat(outs)


def _tile_near(a, Ta, Tb, every):
    """Mask [Ta, Tb]: tiles whose closed longitude arcs meet."""
    if every:
        return torch.ones(Ta, Tb, dtype=torch.bool, device=a)
    s, t = torch.arange(Ta, device=a)[:, None], torch.arange(Tb, device=a)[None, :]
    near = torch.zeros(Ta, Tb, dtype=torch.bool, device=a)
    for turn in (-1, 0, 1):
        b = t + turn * Tb
        near |= (s * Tb <= (b + 1) * Ta) & (b * Ta <= (s + 1) * Tb)
    return near


def _tiled(case, sph, ninv):
    """Dense band blocks under tile adjacency."""
    dev, k, G = ninv.device, case["k"], sph.N // case["k"]

    def rings(g):  # rings of band g in the order of its pixels' rows
        js = list(range(g * k, g * k + k))
        return js if g < G // 2 else js[::-1]

    pairs = {}
    for g in range(G):
        for h in range(max(0, g - 1), min(G, g + 2)):
            for j in rings(g):
                for rho in rings(h):
                    P, Q, gg = sph.constants(j, rho)
                    half = P * Q * gg
                    reach = half if g == h and g in (0, G - 1) else min(half, 4 * k * max(P, Q) + 2 * max(P, Q))
                    pairs[(j, rho)] = reach - (reach - (P + Q)) % 2
    tab = _Table(case, sph, pairs)
    outs, off = [], 0
    for g in range(G):
        n = int(sph.n[g * k])
        K, T = n * k, n // k
        row = torch.arange(K, device=dev)
        M = torch.zeros(K, K, dtype=torch.float64, device=dev)
        for h in range(max(0, g - 1), min(G, g + 2)):
            nh = int(sph.n[h * k])
            near = _tile_near(dev, T, nh // k, g == h and g in (0, G - 1))
            mask = near.repeat_interleave(k, 0).repeat_interleave(k, 1)  # by pixel column
            B = torch.zeros(n, k, nh, k, dtype=torch.float64, device=dev)
            D = torch.zeros(n, k, nh, k, dtype=torch.float64, device=dev) if g == h else None
            c, p = torch.arange(n, device=dev)[:, None], torch.arange(nh, device=dev)[None, :]
            for r, j in enumerate(rings(g)):
                for r2, rho in enumerate(rings(h)):
                    m = pairs[(j, rho)]
                    B[:, r, :, r2] = mask * _kernel_rows(sph, tab.values(tab.b, 0, j, rho, m), j, rho, m, c, p)
                    if g == h:
                        D[:, r, :, r2] = mask * _kernel_rows(sph, tab.values(tab.d, 0, j, rho, m), j, rho, m, c, p)
            B = B.reshape(K, nh * k)
            w = torch.cat([_ring_map(sph, ninv, 0, rho)[:, None] for rho in rings(h)], 1).reshape(-1)
            M += (B * w) @ B.T
            if g == h:
                M += D.reshape(K, K)
        pad = (off + 3) // 4 * 4 - off
        outs += [torch.zeros(pad, dtype=torch.float64, device=dev), M.reshape(-1)]
        off += pad + K * K
    return torch.cat(outs)


def exact(case, seed):
    sph = _Sphere(case)
    kind = case["kind"]
    ninv, x = _maps(case, seed, sph.theta, sph.n, sph.offset, sph.stride, sph.npix)
    if kind == "tiles":
        return {"blocks": _tiled(case, sph, ninv)}
    blocks, size = sph.blocks(case)
    if sum(len(b["near"]) for b in blocks) > 90000:
        return None  # over about 20 seconds
    tab = _ring_table(case, sph, blocks)
    if kind == "convolve":
        return {"g": _convolved(sph, blocks, tab, x)}
    if kind == "coupling":
        return {"blocks": _coupled(case, sph, blocks, tab, ninv)}
    buf = _sampled(case, sph, blocks, size, tab, ninv)
    if kind == "sample":
        return {"blocks": buf}
    if kind == "step":
        return {"blocks": _factored(blocks, buf), "info": None}
    return {"y": _applied(sph, blocks, buf, x)}
