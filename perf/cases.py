"""The work that is timed: what a user of this library has it do, through its public entry points.

A case is one call on one kind of suspension:

  sample   Sampler.sample: one Brownian displacement M^{1/2} z of every particle (FP32 or FP64 context)
  forces   Sampler.sample_with_forces: c_det M F + c_noise M^{1/2} z, the displacement of one Euler-Maruyama step
  bd       Sampler.bd_step: one whole Brownian step in place (repulsion, displacement, new positions)
  batch    BatchSampler.sample: many systems of uneven size in one call
  poly     PolySampler.sample: spheres of several radii

`exact` repeats each of them in plain float64 torch, written from the method's definition (Fiore, Balboa Usabiaga,
Donev & Swan, J. Chem. Phys. 146, 124116 (2017)): the positively split Ewald sum of the periodic
Rotne-Prager-Yamakawa mobility, the real-space part by Lanczos, the wave-space part on an FFT grid.
"""
from __future__ import annotations

import math
import random
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

from paper_1611_09322_gb300 import PSE_FP32, PSE_FP64, BatchSampler, PolySampler, Sampler, workloads

# ---------------------------------------------------------------------------------------------------- the cases


def listed():
    return [
        # one small periodic box, as in method development and in parameter scans: latency of a call
        dict(name="sample-1k", what="sample", kind="hs", N=1000, phi=0.1, xi=0.5, tol=1e-3, M=0, fp64=False),
        # the same box in double precision: reference runs and checks
        dict(name="sample-1k-f64", what="sample", kind="hs", N=1000, phi=0.1, xi=0.5, tol=1e-3, M=0, fp64=True),
        # an ordinary box at the plan's own (odd) grid, the small end of the published timing table
        dict(name="sample-16k", what="sample", kind="hs", N=16001, phi=0.1, xi=0.5, tol=1e-3, M=0, fp64=False),
        # a dense suspension: many neighbours, more Lanczos steps
        dict(name="sample-100k-dense", what="sample", kind="hs", N=100000, phi=0.4, xi=0.6, tol=1e-3, M=0, fp64=False),
        # a colloidal gel: strongly uneven density, empty cells next to full ones
        dict(name="gel-250k", what="sample", kind="gel", N=250047, phi=0.05, xi=0.5, tol=1e-3, M=0, fp64=False),
        # a tight tolerance: wider support, longer cutoff, more Lanczos steps
        dict(name="sample-200k-1e-5", what="sample", kind="hs", N=200000, phi=0.2, xi=0.6, tol=1e-5, M=0, fp64=False),
        # the published size, at the splitting and grid that the timed scan picks for it
        dict(name="sample-1m", what="sample", kind="hs", N=1000000, phi=0.1, xi=0.5178442916, tol=1e-3, M=256, fp64=False),
        # the largest box
        dict(name="sample-4m", what="sample", kind="hs", N=4000000, phi=0.3, xi=0.715, tol=1e-3, M=378, fp64=False),
        # a displacement under given forces (sedimentation, an external field): spreading and both transforms
        dict(name="forces-200k", what="forces", kind="hs", N=200000, phi=0.1, xi=0.5, tol=1e-3, M=0, fp64=False),
        # a step of a Brownian dynamics run of soft spheres with a few overlaps
        dict(name="bd-step-30k", what="bd", kind="soft", N=30001, phi=0.15, xi=0.5, tol=1e-3, M=0, fp64=False),
        # parameter sweeps: many boxes of uneven size and density, half of the dilute ones gels
        dict(name="batch-64", what="batch", nsys=64, spec=1000, n_lo=1000, n_hi=50000, phi_lo=0.05, phi_hi=0.4, tol=1e-3),
        # a binary suspension
        dict(name="poly-100k", what="poly", N=100000, phi=0.1, a1=1.0, a2=0.5, xi=0.5, tol=1e-3, M=0),
    ]


def draw(rng):
    """Another case of the same ranges; sizes are uniform in their logarithm."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    what = rng.choice(["sample", "sample", "sample", "sample", "forces", "bd", "batch", "poly"])
    if what == "batch":
        return dict(what="batch", nsys=rng.randint(3, 64), spec=rng.randrange(1 << 20), n_lo=1000, n_hi=size(4000, 50000),
                    phi_lo=0.05, phi_hi=0.4, tol=1e-3)
    if what == "poly":
        return dict(what="poly", N=size(2000, 300000), phi=round(rng.uniform(0.05, 0.2), 3), a1=1.0,
                    a2=rng.choice([0.5, 0.6, 0.8]), xi=round(rng.uniform(0.45, 0.65), 3), tol=1e-3, M=0)
    fp64 = what == "sample" and rng.random() < 0.2
    kind = "soft" if what == "bd" else rng.choice(["hs", "hs", "gel"])
    tol = 1e-3 if what == "bd" else rng.choice([1e-3, 1e-3, 1e-3, 1e-4, 1e-5])
    hi = 20000 if fp64 else {"sample": 1000000 if tol == 1e-3 else 250000, "forces": 250000, "bd": 50000}[what]
    phi = round(rng.uniform(0.05, 0.15 if kind == "gel" else 0.3 if kind == "soft" else 0.4), 3)
    return dict(what=what, kind=kind, N=size(1000 if tol == 1e-3 else 3000, hi), phi=phi,
                xi=round(rng.uniform(0.5, 0.65), 3), tol=tol, M=0, fp64=fp64)


# ---------------------------------------------------------------------------------------------------- the inputs

def tiles(kind, N, phi):
    """Generating a large dense box or gel sphere by sphere takes minutes, so a box above these sizes is t^3 periodic
    copies of a smaller random one; what a call costs depends on the structure within a few diameters only."""
    most = 2000 if kind == "gel" or phi > 0.3 else 20000 if phi > 0.2 else 150000
    t = 1
    while N / t ** 3 > most:
        t += 1
    return t


def count(kind, N, phi):
    """Particles in the box: N to the next lower multiple of the number of copies."""
    return N // tiles(kind, N, phi) ** 3 * tiles(kind, N, phi) ** 3


def suspension(kind, N, phi, seed):
    """Positions (count, 3) float32 in [0, L) and L. Spheres come in random order, a gel's cluster by cluster."""
    t = tiles(kind, N, phi)
    n0 = N // t ** 3
    if kind == "gel":
        pos, L0, _ = workloads.gel(n0, phi, seed)
    elif kind == "soft":  # placed with a smaller radius: up to 6% overlap at a = 1
        pos, L0, _ = workloads.hard_spheres(n0, phi * 0.97 ** 3, seed, a=0.97)
    else:
        pos, L0, _ = workloads.hard_spheres(n0, phi, seed)
    if t == 1:
        return pos, L0
    s = np.stack(np.meshgrid(*[np.arange(t) * L0] * 3, indexing="ij"), axis=-1).reshape(-1, 1, 3)
    p = (s + pos.astype(np.float64)[None]).reshape(-1, 3)
    if kind != "gel":
        p = p[np.random.default_rng(seed).permutation(p.shape[0])]
    L = t * L0
    p = np.mod(p, L).astype(np.float32)
    p[p >= np.float32(L)] = 0.0
    return p, L


def systems(case, seed):
    """The boxes of a batch: N log-uniform, phi uniform, every second box a gel where it is dilute."""
    r = random.Random(case["spec"])
    spec = []
    for k in range(case["nsys"]):
        N = int(math.exp(r.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]))))
        phi = r.uniform(case["phi_lo"], case["phi_hi"])
        spec.append(("gel" if k % 2 and phi <= 0.2 else "hs", N, phi))
    if seed is None:
        return spec
    with ThreadPoolExecutor(8) as ex:
        return list(ex.map(lambda s: suspension(*s[1], seed * 64 + s[0]), enumerate(spec)))


def inputs(case, seed):
    """Everything a call reads, on the host: made from the case and the seed alone."""
    r = np.random.default_rng(seed + 17)
    if case["what"] == "batch":
        return dict(boxes=systems(case, seed))
    if case["what"] == "poly":
        pos, species, L, _ = workloads.polydisperse(case["N"], case["phi"], seed, radii=(case["a1"], case["a2"]))
        order = r.permutation(pos.shape[0])
        return dict(pos=np.ascontiguousarray(pos[order]), species=np.ascontiguousarray(species[order]), L=L)
    pos, L = suspension(case["kind"], case["N"], case["phi"], seed)
    got = dict(pos=pos.astype(np.float64) if case["fp64"] else pos, L=L)
    if case["what"] in ("forces", "bd"):
        got["F"] = (r.standard_normal(pos.shape) * 0.5 + [0.0, 0.0, -1.0]).astype(np.float32)
    return got


C_DET, C_NOISE = 1e-2, math.sqrt(2 * 1.0 * 1e-2)  # dt = 1e-2, kT = 1
BD = dict(dt=1e-3, kT=1.0, k_rep=100.0)


def batch_grid(L, xi, tol):
    """A batch's grid: the next size of a short list above the plan's, so that boxes share their transforms."""
    M = make_plan(L, 1.0, xi, tol, 0).M
    return next(m for m in (20, 24, 32, 40, 48, 64, 80, 96, 112, 128, 160, 192, 256) if m >= M)


def prepare(case, seed):
    x = inputs(case, seed)
    dev = lambda v: torch.from_numpy(v).cuda()  # noqa: E731
    st = dict(what=case["what"], seed=seed)
    if case["what"] == "batch":
        Ls = [L for _, L in x["boxes"]]
        st["offsets"] = np.cumsum([0] + [p.shape[0] for p, _ in x["boxes"]])
        st["pos"] = dev(np.concatenate([p for p, _ in x["boxes"]]))
        st["s"] = BatchSampler(Ls, 1.0, params=[dict(xi=0.5, tol=case["tol"], grid_M=batch_grid(L, 0.5, case["tol"]))
                                                for L in Ls])
        return st
    st["pos"] = dev(x["pos"])
    if case["what"] == "poly":
        st["species"] = dev(x["species"])
        st["s"] = PolySampler(x["L"], (case["a1"], case["a2"]), xi=case["xi"], tol=case["tol"], grid_M=case["M"])
        return st
    st["s"] = Sampler(x["L"], 1.0, xi=case["xi"], tol=case["tol"], grid_M=case["M"],
                      precision=PSE_FP64 if case["fp64"] else PSE_FP32)
    if "F" in x:
        st["F"] = dev(x["F"])
    return st


def run(state):
    s, pos, what = state["s"], state["pos"], state["what"]
    if what == "sample":
        return s.sample(pos, state["seed"], 0)
    if what == "forces":
        return s.sample_with_forces(pos, state["F"], state["seed"], 0, C_DET, C_NOISE)
    if what == "bd":  # the caller keeps the frame that the step starts from
        return s.bd_step(pos.clone(), state["seed"], 0, f_ext=state["F"], **BD)
    if what == "poly":
        return s.sample(pos, state["species"], state["seed"], 0)
    return s.sample(pos, state["offsets"], state["seed"], 0)


# ---------------------------------------------------------------------------------------------------- work and tolerance

def work(case):
    """Positions (and forces, species) read and displacements written once; each velocity grid written by the inverse
    transform and read by the interpolation; the positions and vectors of four Lanczos products. Operations: the
    transforms, the P^3 interpolation (and spreading), the pair blocks within the cutoff."""
    if case["what"] == "batch":
        both = [_work(n, phi, 0.5, case["tol"], batch_grid(workloads.box_length(n, phi), 0.5, case["tol"]), 4, 1, False)
                for n, phi in ((count(*s), s[2]) for s in systems(case, None))]
        return {k: sum(b[k] for b in both) for k in ("bytes", "flops")}
    if case["what"] == "poly":
        v3 = 0.5 * (case["a1"] ** 3 + case["a2"] ** 3)
        return _work(case["N"], case["phi"], case["xi"], case["tol"], 0, 4, 2, False, v3, min(case["a1"], case["a2"]))
    n = count(case["kind"], case["N"], case["phi"])
    return _work(n, case["phi"], case["xi"], case["tol"], case["M"], 8 if case["fp64"] else 4, 1, case["what"] != "sample")


def _work(N, phi, xi, tol, M, size, grids, forces, v3=1.0, a=1.0):
    L = (N * 4.0 / 3.0 * math.pi * v3 / phi) ** (1.0 / 3.0)
    p = make_plan(L, a, xi, tol, M)
    pairs = N * N / L ** 3 * 4.0 / 3.0 * math.pi * p.rc ** 3
    steps, ways = 4, 2 if forces else 1
    fft = 3 * 2.5 * p.M ** 3 * math.log2(p.M ** 3)
    return {"bytes": size * (6 * N + 6 * grids * ways * p.M ** 3 + steps * 9 * N + (3 * N if forces else 0)),
            "flops": grids * ways * fft + ways * N * 6 * p.P ** 3 + (steps + ways - 1) * pairs * 30}


def tolerance(case):
    """About four times the distance from `exact` over the listed and some drawn cases: FP32 displacements 3.4e-7 to
    9.8e-7 (largest single value 9e-5 of the root mean square, at 4e6 particles), FP64 5e-14, new positions 2.6e-8."""
    if case.get("fp64"):
        return {"rel": 4e-13}
    if case["what"] == "bd":
        return {"rel": 1.2e-7, "max": 6e-7}
    return {"rel": 4e-6, "max": 4e-4}


# ---------------------------------------------------------------------------------------------------- the plan, in plain Python

class Plan:
    pass


def make_plan(L, a, xi, tol, M):
    """Cutoffs, grid and Gaussian of one box (the paper's Sec. II C)."""
    p = Plan()
    p.L, p.a, p.xi, p.tol = L, a, xi, tol
    p.rc = math.sqrt(math.log(1.0 / tol)) / xi

    def left(k):
        return (4.0 / k * math.exp(-k * k / (4 * xi * xi)) - math.sqrt(math.pi) / xi * math.erfc(k / (2 * xi))) / (2 * math.pi * a)

    def error(P, m):
        return math.exp(-math.pi ** 2 * P * P / (2 * m * m)) + math.erfc(m / math.sqrt(2.0))

    def slope(P, m):
        c = math.pi ** 2 * P * P / 2.0
        return math.exp(-c / (m * m)) * 2 * c / m ** 3 - math.sqrt(2 / math.pi) * math.exp(-m * m / 2)

    def root(lo, hi, above):
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            lo, hi = (mid, hi) if above(mid) else (lo, mid)
        return hi

    def smooth(n):
        for q in (2, 3, 5, 7):
            while n % q == 0:
                n //= q
        return n == 1

    p.P = 3
    while True:
        lo, hi = 0.5, 2.0 * p.P
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            lo, hi = (mid, hi) if slope(p.P, mid) < 0 else (lo, mid)
        p.m = 0.5 * (lo + hi)
        if error(p.P, p.m) <= tol:
            break
        p.P += 1
    if M <= 0:
        top = 1.0
        while left(top) > tol:
            top *= 2.0
        kc = root(1e-6, top, lambda k: left(k) > tol)
        M = max(int(math.ceil(kc * L / math.pi - 1e-9)), p.P + 1, 4)
        while not smooth(M) or (p.P * (L / M) * xi / p.m) ** 2 > 1.0:
            M += 1
    p.M, p.h = M, L / M
    p.eta = (p.P * p.h * xi / p.m) ** 2
    return p


# ---------------------------------------------------------------------------------------------------- float64

MASK = 0xFFFFFFFF


def normals(element, stream, seed, sample):
    """Four N(0,1) per element: Philox4x32-10 (Salmon et al., SC'11), key = seed, counter = (element, stream, sample),
    23-bit uniforms, Box-Muller. 32-bit words in int64; a product's upper word survives the wrap to 64 bits."""
    c0 = element & MASK
    c1 = torch.full_like(c0, stream)
    c2 = torch.full_like(c0, sample & MASK)
    c3 = torch.full_like(c0, sample >> 32)
    k0, k1 = seed & MASK, seed >> 32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & MASK) ^ c1 ^ k0, p1 & MASK, ((p0 >> 32) & MASK) ^ c3 ^ k1, p0 & MASK
        k0, k1 = (k0 + 0x9E3779B9) & MASK, (k1 + 0xBB67AE85) & MASK
    u = [((c >> 9).double() + 0.5) * 2.0 ** -23 for c in (c0, c1, c2, c3)]
    ra, rc = torch.sqrt(-2.0 * torch.log(u[0])), torch.sqrt(-2.0 * torch.log(u[2]))
    return (ra * torch.cos(2 * math.pi * u[1]), ra * torch.sin(2 * math.pi * u[1]),
            rc * torch.cos(2 * math.pi * u[3]), rc * torch.sin(2 * math.pi * u[3]))


def free_pair(r, ai, aj):
    """Rotne-Prager-Yamakawa tensor of two spheres, A (I - rr) + (A + B) rr, as (F, G)."""
    s2, d2 = ai * ai + aj * aj, (ai - aj) ** 2
    far, inner = r > ai + aj, r <= (ai - aj).abs()
    A = torch.where(far, (1 + s2 / (3 * r * r)) / (8 * math.pi * r),
                    (16 * r ** 3 * (ai + aj) - (d2 + 3 * r * r) ** 2) / (32 * r ** 3) / (6 * math.pi * ai * aj))
    B = torch.where(far, (1 - s2 / (r * r)) / (8 * math.pi * r), 3 * (d2 - r * r) ** 2 / (32 * r ** 3) / (6 * math.pi * ai * aj))
    return torch.where(inner, 1 / (6 * math.pi * torch.maximum(ai, aj)), A), torch.where(inner, 0 * A, A) + torch.where(inner, 0 * B, B)


def wave_pair(r, xi, ai, aj):
    """The part of a pair that the wave sum carries: the k-integral weighted with H = (1 + q) e^-q, q = k^2/4 xi^2."""
    t, w = np.polynomial.legendre.leggauss(160)
    k = torch.tensor(8.0 * xi * (t + 1.0), device=r.device)
    w = torch.tensor(8.0 * xi * w, device=r.device)
    q = k * k / (4 * xi * xi)
    sinc = lambda x: torch.sinc(x / math.pi)  # noqa: E731
    F, G = torch.empty_like(r), torch.empty_like(r)
    step = 1 << 18
    for s in range(0, r.numel(), step):
        e = slice(s, s + step)
        base = (1 + q) * torch.exp(-q) * w * sinc(ai[e, None] * k) * sinc(aj[e, None] * k)
        x = r[e, None] * k
        xs = torch.where(x < 2e-2, torch.ones_like(x), x)
        sn, cs = torch.sin(xs), torch.cos(xs)
        kF = torch.where(x < 2e-2, 2 / 3 - 2 * x * x / 15 + x ** 4 / 140, (xs * cs + (xs * xs - 1) * sn) / xs ** 3)
        kG = torch.where(x < 2e-2, 1 / 3 - x * x / 30 + x ** 4 / 840, (sn - xs * cs) / xs ** 3)
        F[e], G[e] = (kF * base).sum(1) / (2 * math.pi ** 2), (kG * base).sum(1) / math.pi ** 2
    return F, G


def real_pair(r, xi, ai, aj):
    """Real-space pair scalars: the free tensor less what the wave sum carries."""
    Ff, Gf = free_pair(r, ai, aj)
    if r.numel() < 4096:
        Fw, Gw = wave_pair(r, xi, ai, aj)
        return Ff - Fw, Gf - Gw
    # the wave part is analytic in r, with variations of length 1/xi and up: one Chebyshev series of degree 63 per pair
    # of radii on [0, rmax] holds it to rounding
    rmax = float(r.max()) * (1 + 1e-12)
    n = 64
    th = (torch.arange(n, device=r.device, dtype=torch.float64) + 0.5) * math.pi / n
    nodes = 0.5 * rmax * (torch.cos(th) + 1)
    Fw, Gw = torch.empty_like(r), torch.empty_like(r)
    T = torch.cos(th[None] * torch.arange(n, device=r.device, dtype=torch.float64)[:, None])
    for x in torch.unique(ai).tolist():
        for y in torch.unique(aj).tolist():
            f, g = wave_pair(nodes, xi, torch.full_like(nodes, x), torch.full_like(nodes, y))
            cf, cg = (T @ f) * (2.0 / n), (T @ g) * (2.0 / n)
            cf[0] *= 0.5
            cg[0] *= 0.5
            at = torch.nonzero((ai == x) & (aj == y)).flatten()
            s = 2 * r[at] / rmax - 1
            for c, out in ((cf, Fw), (cg, Gw)):
                c = c.tolist()
                b1, b2 = torch.zeros_like(s), torch.zeros_like(s)
                for j in range(n - 1, 0, -1):
                    b1, b2 = 2 * s * b1 - b2 + c[j], b1
                out[at] = s * b1 - b2 + c[0]
    return Ff - Fw, Gf - Gw


def pairs(p, L, rc):
    """Directed pairs (i, j, x_i - x_j) within rc, nearest image, by cells of side >= rc."""
    N = p.shape[0]
    nc = max(1, min(200, int(L / rc)))
    if nc < 3:
        d = p[:, None] - p[None]
        d -= L * torch.round(d / L)
        i, j = torch.nonzero((d.square().sum(-1) < rc * rc) & ~torch.eye(N, dtype=torch.bool, device=p.device), as_tuple=True)
        return i, j, d[i, j]
    c = torch.clamp((p * (nc / L)).long(), max=nc - 1)
    cell = (c[:, 0] * nc + c[:, 1]) * nc + c[:, 2]
    order = torch.argsort(cell)
    number = torch.bincount(cell, minlength=nc ** 3)
    start = torch.cumsum(number, 0) - number
    most = int(number.max())
    step = max(1, (1 << 26) // most)
    got = []
    for ox in (-1, 0, 1):
        for oy in (-1, 0, 1):
            for oz in (-1, 0, 1):
                for s in range(0, N, step):
                    i = torch.arange(s, min(N, s + step), device=p.device)
                    b = c[i] + torch.tensor([ox, oy, oz], device=p.device)
                    b = torch.remainder(b, nc)
                    b = (b[:, 0] * nc + b[:, 1]) * nc + b[:, 2]
                    k = torch.arange(most, device=p.device)
                    a, k = torch.nonzero(k[None] < number[b][:, None], as_tuple=True)
                    j, i = order[start[b[a]] + k], i[a]
                    d = p[i] - p[j]
                    d -= L * torch.round(d / L)
                    keep = (d.square().sum(1) < rc * rc) & (i != j)
                    got.append((i[keep], j[keep], d[keep]))
    return tuple(torch.cat([g[n] for g in got]) for n in range(3))


class Near:
    """M_r as a product, from its pairs."""

    def __init__(self, p, radii, plan):
        self.i, self.j, d = pairs(p, plan.L, plan.rc)
        r = d.norm(dim=1)
        F, G = real_pair(r, plan.xi, radii[self.i], radii[self.j])
        self.rh, self.F, self.GF = d / r[:, None], F, G - F
        self.d = d
        one = {}
        for a in torch.unique(radii).tolist():
            t = torch.tensor([a], dtype=torch.float64, device=p.device)
            one[a] = 1 / (6 * math.pi * a) - float(wave_pair(0 * t, plan.xi, t, t)[0])
        self.own = torch.empty_like(radii)
        for a, v in one.items():
            self.own[radii == a] = v

    def __call__(self, v):
        out = self.own[:, None] * v
        step = 1 << 25
        for s in range(0, self.i.numel(), step):
            e = slice(s, s + step)
            vj, rh = v[self.j[e]], self.rh[e]
            out.index_add_(0, self.i[e], self.F[e, None] * vj + (self.GF[e] * (rh * vj).sum(1))[:, None] * rh)
        return out


def lanczos(A, z, tol):
    """A^{1/2} z: x_j = |z| V_j T_j^{1/2} e_1, to the first j >= 2 with |x_j - x_{j-1}| < tol |x_j|."""
    nz = float(z.norm())
    V, al, be, before = [z / nz], [], [], None
    for j in range(1, 101):
        w = A(V[-1])
        if j > 1:
            w -= be[-1] * V[-2]
        al.append(float((w * V[-1]).sum()))
        w -= al[-1] * V[-1]
        be.append(float(w.norm()))
        lam, Q = np.linalg.eigh(np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1))
        y = Q @ (np.sqrt(lam) * Q[0])
        if before is not None and np.linalg.norm(y - np.append(before, 0.0)) < tol * np.linalg.norm(y):
            break
        before = y
        V.append(w / be[-1])
    return nz * sum(float(c) * v for c, v in zip(y, V))


def noise_and_modes(plan, a, seed, system, dev, det=None, c_det=0.0, c_noise=1.0):
    """The half spectrum (3, M, M, M//2+1) of the velocity grid: c_noise times the scaled projected noise, plus c_det
    times the mode factor on a spread force's transform `det`."""
    M, L = plan.M, plan.L
    H = M // 2 + 1
    n = torch.arange(M, device=dev)
    n = torch.where(n > M // 2, n - M, n)
    nz = torch.arange(H, device=dev)
    kx, ky, kz = (n.double() * (2 * math.pi / L))[:, None, None], (n.double() * (2 * math.pi / L))[None, :, None], (nz.double() * (2 * math.pi / L))[None, None]
    k2 = kx * kx + ky * ky + kz * kz
    k2[0, 0, 0] = 1.0
    k = torch.sqrt(k2)
    scale = torch.sinc(k * a / math.pi) / k * torch.sqrt(1 + k2 / (4 * plan.xi ** 2)) * torch.exp(-(1 - plan.eta) * k2 / (8 * plan.xi ** 2)) / math.sqrt(L ** 3)
    scale[0, 0, 0] = 0.0
    if M % 2 == 0:
        scale[M // 2], scale[:, M // 2], scale[:, :, M // 2] = 0.0, 0.0, 0.0
    if c_noise:
        q = torch.arange(M * M * H, device=dev)
        a4, b4 = normals(2 * q, 2 * system + 1, seed, 0), normals(2 * q + 1, 2 * system + 1, seed, 0)
        w = torch.stack([torch.complex(a4[0], a4[1]), torch.complex(a4[2], a4[3]), torch.complex(b4[0], b4[1])]).reshape(3, M, M, H) / math.sqrt(2.0)
        del a4, b4
        first = (n[None, :] > 0) | ((n[None, :] == 0) & (n[:, None] > 0))  # of each pair {k, -k} in the plane nz = 0
        w0 = w[:, :, :, 0] * first
        w[:, :, :, 0] = w0 + torch.roll(torch.flip(w0, (1, 2)), (1, 1), (1, 2)).conj()
        w *= c_noise * scale
    else:
        w = torch.zeros((3, M, M, H), dtype=torch.complex128, device=dev)
    if det is not None:
        w += c_det * plan.h ** 3 * scale * scale * det
    dot = (kx * w[0] + ky * w[1] + kz * w[2]) / k2
    return torch.stack([w[0] - kx * dot, w[1] - ky * dot, w[2] - kz * dot])


def support(p, plan):
    """Node indices and Gaussian weights (N, P) of each particle along each axis."""
    c = 2 * plan.xi ** 2 / plan.eta
    at, wt = [], []
    for d in range(3):
        s = p[:, d] * plan.M / plan.L
        g = (torch.floor(s - plan.P / 2.0).long() + 1)[:, None] + torch.arange(plan.P, device=p.device)
        wt.append(torch.exp(-c * ((s[:, None] - g) * plan.h) ** 2) * math.sqrt(c / math.pi))
        at.append(torch.remainder(g, plan.M))
    return at, wt


def from_grid(spec, p, plan):
    M = plan.M
    v = torch.stack([torch.fft.irfftn(spec[d], s=(M, M, M), norm="forward").reshape(-1) for d in range(3)], dim=1)
    at, wt = support(p, plan)
    out = torch.zeros_like(p)
    for x in range(plan.P):
        for y in range(plan.P):
            for z in range(plan.P):
                node = (at[0][:, x] * M + at[1][:, y]) * M + at[2][:, z]
                out += (wt[0][:, x] * wt[1][:, y] * wt[2][:, z])[:, None] * v[node]
    return out * plan.h ** 3


def to_grid(F, p, plan):
    M = plan.M
    at, wt = support(p, plan)
    s = torch.zeros((M ** 3, 3), dtype=torch.float64, device=p.device)
    for x in range(plan.P):
        for y in range(plan.P):
            for z in range(plan.P):
                s.index_add_(0, (at[0][:, x] * M + at[1][:, y]) * M + at[2][:, z], (wt[0][:, x] * wt[1][:, y] * wt[2][:, z])[:, None] * F)
    return torch.stack([torch.fft.rfftn(s[:, d].reshape(M, M, M)) for d in range(3)])


def displacement(p, plan, seed, system=0, F=None, c_det=0.0, c_noise=1.0, near=None):
    """c_det M F + c_noise M^{1/2} z of equal spheres."""
    near = Near(p, torch.full((p.shape[0],), plan.a, dtype=torch.float64, device=p.device), plan) if near is None else near
    z = torch.stack(normals(torch.arange(p.shape[0], device=p.device), 2 * system, seed, 0)[:3], dim=1)
    out = c_noise * lanczos(near, z, plan.tol)
    det = None
    if F is not None:
        out += c_det * near(F)
        det = to_grid(F, p, plan)
    del near
    return out + from_grid(noise_and_modes(plan, plan.a, seed, system, p.device, det, c_det, c_noise), p, plan)


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    x = inputs(case, seed)
    up = lambda v: torch.from_numpy(np.asarray(v, dtype=np.float64)).to(dev)  # noqa: E731
    if case["what"] == "batch":
        return torch.cat([displacement(up(p), make_plan(L, 1.0, 0.5, case["tol"], batch_grid(L, 0.5, case["tol"])), seed, k)
                          for k, (p, L) in enumerate(x["boxes"])])
    p, L = up(x["pos"]), x["L"]
    if case["what"] == "poly":
        plan = make_plan(L, min(case["a1"], case["a2"]), case["xi"], case["tol"], case["M"])
        species = torch.from_numpy(x["species"]).to(dev).long()
        radii = torch.tensor([case["a1"], case["a2"]], dtype=torch.float64, device=dev)
        z = torch.stack(normals(torch.arange(p.shape[0], device=dev), 0, seed, 0)[:3], dim=1)
        out = lanczos(Near(p, radii[species], plan), z, plan.tol)
        for s in range(2):
            out[species == s] += from_grid(noise_and_modes(plan, float(radii[s]), seed, 0, dev), p[species == s], plan)
        return out
    plan = make_plan(L, 1.0, case["xi"], case["tol"], case["M"])
    if case["what"] == "sample":
        return displacement(p, plan, seed)
    F = up(x["F"])
    if case["what"] == "forces":
        return displacement(p, plan, seed, 0, F, C_DET, C_NOISE)
    near = Near(p, torch.ones(p.shape[0], dtype=torch.float64, device=dev), plan)
    r = near.d.norm(dim=1)
    push = torch.nonzero(r < 2.0).flatten()
    F = F.index_add(0, near.i[push], (BD["k_rep"] * (2.0 - r[push]) / r[push])[:, None] * near.d[push])
    return torch.remainder(p + displacement(p, plan, seed, 0, F, BD["dt"], math.sqrt(2 * BD["kT"] * BD["dt"]), near), L)
