"""Workloads of the harmonic 3PCF estimator, as a user's program runs them.

Every case goes through the public entry points (``tpcf.Plan``, ``tpcf.ZetaFn``,
``tpcf.Batch``, ``Plan.run_host_into``).  A case holds its kind, its sizes and its seed-free
options; ``prepare`` paints the inputs on the GPU from the seed and builds the plan
that a program keeps.  ``exact`` is the estimator in 64 bits, written with torch alone.

The data vector is kept in single precision, as its accuracy is: the library sums fp32
moments (stated accuracy 1e-5 of the largest entry per multipole, measured 4e-8 to 5e-7
against ``exact`` on these cases), and the digits of the 64-bit container beyond that
depend on the order of the sums and differ between two runs on the same input.
"""
import math

import numpy as np
import torch

from paper_2408_16847_gb300 import tpcf

DEV = "cuda"


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the smallest call in use: one likelihood-gradient step on a coarse map (the
        # library's smoke size); latency and launches count
        dict(name="map16_step", kind="map_step", nside=16, k=6, m=6, lo=1.0, hi=12.0, log=True, w="unit",
             opt="default", a=0.0, b=1.0),
        # plain forward of a small full-sky map: one mock of a large ensemble
        dict(name="map64_fwd", kind="map_fwd", nside=64, k=10, m=8, lo=0.5, hi=10.0, log=False, w="unit",
             opt="default", a=0.0, b=1.0),
        # end to end from pinned host buffers: host map in, estimate and gradient out
        dict(name="map256_host", kind="map_host", nside=256, k=16, m=8, lo=0.2, hi=4.0, log=True, w="unit",
             opt="default", a=0.0, b=1.0),
        # an ordinary full-sky map, short rows of neighbours per ring and bin
        dict(name="map512_fwd", kind="map_fwd", nside=512, k=20, m=10, lo=0.1, hi=2.0, log=True, w="unit",
             opt="default", a=0.0, b=1.0),
        # masked survey map with the gradient of a loss (field-level inference)
        dict(name="map1024_masked_step", kind="map_step", nside=1024, k=20, m=10, lo=0.2, hi=3.0, log=True,
             w="mask", opt="default", a=0.0, b=1.0),
        # one rank's pivots of the Nside 4096 map in the equatorial belt, with gradient
        dict(name="map4096_belt_step", kind="map_step", nside=4096, k=20, m=10, lo=0.1, hi=2.0, log=True,
             w="unit", opt="default", a=0.5, b=0.5016),
        # one rank's pivots of the Nside 4096 map in the polar cap (a third of the sky)
        dict(name="map4096_cap_fwd", kind="map_fwd", nside=4096, k=20, m=10, lo=0.1, hi=2.0, log=True,
             w="unit", opt="default", a=0.06, b=0.0616),
        # fast approximate mode (shared neighbour lists) on a full map
        dict(name="map1024_grouped", kind="map_grouped", nside=1024, k=20, m=8, lo=0.13, hi=3.33, log=True,
             w="unit", opt="default", a=0.0, b=1.0, group=15),
        # three tomographic fields, cross estimate with their own weights
        dict(name="map256_multi", kind="map_multi", nside=256, k=12, m=8, lo=0.3, hi=4.0, log=True, w="random",
             opt="default", a=0.0, b=1.0),
        # mocks of mixed resolution, bins and multipoles, forward + adjoint in one graph
        dict(name="batch_mixed", kind="batch", maps=12, nside=64, levels=3, k=8, m=6, lo=0.5, hi=4.0),
        # survey catalogue: clustered data with weights, and three times as many randoms
        dict(name="catalog_2e6_fwd", kind="cat_fwd", n=2_000_000, randoms=6_000_000, parents=10_000, k=16, m=10,
             lo=0.1, hi=2.0, log=False, opt="default"),
        # a small catalogue with the gradient
        dict(name="catalog_5e4_step", kind="cat_step", n=20_000, randoms=30_000, parents=200, k=12, m=8, lo=0.2,
             hi=4.0, log=False, opt="default"),
    ]


# Share of the drawn cases by kind.
KINDS = ("map_fwd", "map_fwd", "map_step", "map_step", "map_host", "map_grouped", "map_multi", "batch", "cat_fwd",
         "cat_step")


def draw(rng):
    kind = rng.choice(KINDS)
    k = rng.randint(1, 24)
    m = rng.randint(0, 12) if rng.random() < 0.85 else rng.randint(13, 16)
    if kind == "batch":
        return dict(kind=kind, maps=rng.randint(2, 14), nside=rng.randint(16, 72), levels=rng.randint(1, 3),
                    k=rng.randint(4, 16), m=rng.randint(2, 8), lo=rng.uniform(0.4, 1.0), hi=rng.uniform(2.0, 4.0))
    if kind.startswith("cat"):
        n = int(round(math.exp(rng.uniform(math.log(2_000), math.log(600_000 if kind == "cat_fwd" else 150_000)))))
        # mean neighbours of a point between a few and a few hundred
        hi = min(20.0, math.degrees(2.0 * math.sqrt(math.exp(rng.uniform(math.log(8), math.log(500))) / n)))
        opt = rng.choice(["default", "default", "subtract", "bin_mean", "pivot_total"]) if kind == "cat_fwd" else "default"
        return dict(kind=kind, n=n, randoms=rng.randint(0, 2) * n, parents=max(20, n // rng.randint(50, 300)), k=k, m=m,
                    lo=hi / rng.uniform(8.0, 25.0), hi=hi, log=rng.random() < 0.5, opt=opt)
    top = dict(map_fwd=900, map_step=500, map_host=400, map_grouped=1200, map_multi=260)[kind]
    nside = int(round(math.exp(rng.uniform(math.log(8), math.log(top)))))
    pix = math.degrees(math.sqrt(math.pi / 3.0) / nside)
    hi = min(40.0, pix * math.exp(rng.uniform(math.log(6.0), math.log(45.0 if nside < 500 else 30.0))))
    lo = max(0.7 * pix, hi / rng.uniform(8.0, 25.0))
    opt = "default"
    if kind == "map_fwd":
        opt = rng.choice(["default", "default", "subtract", "tc", "bin_mean", "pivot_total"])
    elif kind == "map_step":
        opt = rng.choice(["default", "default", "subtract"])
    elif kind == "map_multi":
        m, k = min(m, 10), min(k, 16)
    a, b = 0.0, 1.0
    if kind in ("map_fwd", "map_step", "map_grouped") and rng.random() < 0.35:
        a = rng.uniform(0.0, 0.7)
        b = a + rng.uniform(0.05, 0.3)
    c = dict(kind=kind, nside=nside, k=k, m=m, lo=lo, hi=hi, log=rng.random() < 0.5,
             w=rng.choice(["unit", "unit", "mask", "random"]), opt=opt, a=a, b=b)
    if kind == "map_grouped":
        c["group"] = rng.randint(2, 30)
    return c


# ---------------------------------------------------------------- the geometry

def edges_of(case):
    lo, hi, k = case["lo"], case["hi"], case["k"]
    return lo * (hi / lo) ** (np.arange(k + 1) / k) if case.get("log", True) else np.linspace(lo, hi, k + 1)


def ring_table(nside):
    """(z, sin theta, pixels, shift, first pixel) of every HEALPix ring, float64 / int64 on the host;
    pixel p of a ring sits at longitude pi (2 p + shift) / pixels."""
    r = np.arange(1, 4 * nside, dtype=np.int64)
    cap = np.minimum(r, 4 * nside - r)
    north = cap < nside
    t = cap.astype(np.float64) ** 2 / (3.0 * nside * nside)
    belt = (4 * nside - 2 * r).astype(np.float64) / (3.0 * nside)
    z = np.where(north, np.where(r < nside, 1.0 - t, t - 1.0), belt)
    s = np.where(north, np.sqrt(t * (2.0 - t)), np.sqrt(np.maximum(0.0, (1.0 - belt) * (1.0 + belt))))
    n = 4 * np.minimum(cap, nside)
    shift = np.where(north, 1, (r - nside + 1) & 1)
    first = np.concatenate([[0], np.cumsum(n)[:-1]])
    return z, s, n, shift, first


def directions(nside):
    """Pixel centres (x, y, z) of the map, float32 on the GPU."""
    z, s, n, shift, first = (torch.from_numpy(v).to(DEV) for v in ring_table(nside))
    p = torch.arange(12 * nside * nside, device=DEV, dtype=torch.int32)
    rep = lambda v: torch.repeat_interleave(v, n)  # noqa: E731
    phi = (2.0 * (p - rep(first.int())) + rep(shift.float())) * rep(torch.pi / n.float())
    st = rep(s.float())
    return st * torch.cos(phi), st * torch.sin(phi), rep(z.float())


# ------------------------------------------------------------------- the inputs

def field(nside, g, noise=0.05):
    """A mean-subtracted lognormal field with structure from the pixel to tens of degrees, and
    white noise: the one-point shape of a convergence map."""
    x, y, z = directions(nside)
    v = torch.zeros_like(x)
    for i in range(10):
        u = torch.randn(3, generator=g, device=DEV)
        kappa = min(3.0 * 2.1 ** i, 0.7 * nside)
        u = u / u.norm() * kappa
        v += (0.9 ** i) * torch.cos(x * u[0] + y * u[1] + z * u[2] + 6.28 * torch.rand(1, generator=g, device=DEV))
    v = torch.exp(0.5 * v)
    v += noise * torch.randn(v.shape, generator=g, device=DEV)
    return v - v.mean()


def map_weights(kind, nside, g):
    npix = 12 * nside * nside
    if kind == "unit":
        return torch.ones(npix, device=DEV)
    if kind == "random":
        return 0.5 + torch.rand(npix, generator=g, device=DEV)
    z, _, n, _, _ = ring_table(nside)  # the galactic cut |b| < 20 deg
    keep = torch.from_numpy((np.abs(z) >= math.sin(math.radians(20.0))).astype(np.float32)).to(DEV)
    return torch.repeat_interleave(keep, torch.from_numpy(n).to(DEV))


def catalog_points(case, g):
    """Clustered data points, then uniform randoms; delta = 1 / -alpha, data weights in [0.5, 1.5)."""
    n, nr = case["n"], case["randoms"]
    unit = lambda v: v / v.norm(dim=1, keepdim=True)  # noqa: E731
    normal = lambda *s: torch.randn(*s, generator=g, device=DEV, dtype=torch.float64)  # noqa: E731
    parents = unit(normal(case["parents"], 3))
    pick = torch.randint(0, case["parents"], (n,), generator=g, device=DEV)
    sigma = 0.3 * math.radians(case["hi"]) / 2.0 + 0.1 * math.sqrt(4.0 / case["parents"])
    data = unit(parents[pick] + sigma * normal(n, 3))
    w = 0.5 + torch.rand(n, generator=g, device=DEV)
    if not nr:
        return data, torch.randn(n, generator=g, device=DEV), w
    alpha = float(w.double().sum()) / nr
    xyz = torch.cat([data, unit(normal(nr, 3))]).contiguous()
    delta = torch.cat([torch.ones(n, device=DEV), torch.full((nr,), -alpha, device=DEV)])
    return xyz, delta, torch.cat([w, torch.ones(nr, device=DEV)])


def cotangent(case, g):
    c = torch.zeros(case["m"] + 1, case["k"], case["k"], 2, dtype=torch.float64, device=DEV)
    c[..., 0] = torch.randn(c.shape[:-1], generator=g, device=DEV, dtype=torch.float64)
    return c


def pivots_of(case, npix):
    lo, hi = int(round(case.get("a", 0.0) * npix)), int(round(case.get("b", 1.0) * npix))
    return lo, max(lo + 1, min(npix, hi))


def batch_members(case):
    """Plain map cases of the batch's members: mixed resolution, bins, spacing and multipoles."""
    out = []
    for i in range(case["maps"]):
        out.append(dict(kind="map_member", nside=case["nside"] * 2 ** (i % case["levels"]), k=case["k"] + (5 * i) % 7,
                        m=case["m"] + (3 * i) % 5, lo=case["lo"], hi=case["hi"], log=i % 2 == 0, w="unit",
                        opt="default"))
    return out


def with_gradient(kind):
    return kind.endswith("_step") or kind in ("map_host", "map_member")


def plan_options(opt):
    return {"default": {}, "subtract": {"self_pairs": "subtract"}, "tc": {"contract": "tc"},
            "bin_mean": {"norm": "bin_mean"}, "pivot_total": {"norm": "pivot_total"}}[opt]


def inputs(case, seed):
    """The case's arrays alone (no plan)."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    kind = case["kind"]
    if kind.startswith("cat"):
        xyz, delta, w = catalog_points(case, g)
        return dict(xyz=xyz, delta=delta, w=w, cot=cotangent(case, g))
    if kind == "batch":
        return dict(members=[inputs(c, seed * 1000 + i) for i, c in enumerate(batch_members(case))])
    if kind == "map_multi":
        return dict(fields=[(field(case["nside"], g), map_weights(case["w"], case["nside"], g)) for _ in range(3)])
    return dict(delta=field(case["nside"], g), w=map_weights(case["w"], case["nside"], g), cot=cotangent(case, g))


def prepare(case, seed):
    s = inputs(case, seed)
    s["case"] = case
    kind = case["kind"]
    if kind == "batch":
        cases = batch_members(case)
        s["plans"] = [tpcf.Plan.map(c["nside"], edges_of(c), c["m"]) for c in cases]
        new = lambda *shape: torch.empty(*shape, dtype=torch.float64, device=DEV)  # noqa: E731
        s["zeta"] = [new(*p.zeta_shape()) for p in s["plans"]]
        s["norm"] = [new(p.K, p.K) for p in s["plans"]]
        s["grad"] = [torch.empty_like(x["delta"]) for x in s["members"]]
        s["batch"] = tpcf.Batch(s["plans"], [x["delta"] for x in s["members"]], [x["w"] for x in s["members"]],
                                s["zeta"], s["norm"], [x["cot"] for x in s["members"]], s["grad"])
        return s
    if kind.startswith("cat"):
        s["plan"] = tpcf.Plan.catalog(s["xyz"], edges_of(case), case["m"], **plan_options(case["opt"]))
    else:
        s["plan"] = tpcf.Plan.map(case["nside"], edges_of(case), case["m"], **plan_options(case["opt"]))
        s["range"] = pivots_of(case, s["plan"].npoints)
    if kind == "map_host":  # the program's own pinned buffers
        pin = lambda t: t.cpu().pin_memory()  # noqa: E731
        p = s["plan"]
        s["host"] = [pin(s.pop(n)) for n in ("delta", "w", "cot")]
        s["out"] = [pin(torch.zeros(p.zeta_shape(), dtype=torch.float64)),
                    pin(torch.zeros(p.K, p.K, dtype=torch.float64)), pin(torch.zeros(p.npoints))]
    elif kind.endswith("_step"):
        s["delta"].requires_grad_(True)
    return s


# ------------------------------------------------------------------- one pass

def run(state):
    kind = state["case"]["kind"]
    if kind == "batch":
        state["batch"].launch()
        return {"zeta": [z.float() for z in state["zeta"]], "norm": [n.float() for n in state["norm"]],
                "grad": state["grad"]}
    plan = state["plan"]
    if kind == "map_host":
        zeta, norm, grad = plan.run_host_into(*state["host"], out=state["out"])
        return {"zeta": zeta.float(), "norm": norm.float(), "grad": grad}
    if kind.endswith("_step"):
        lo, hi = state.get("range", (0, plan.npoints))
        zeta = tpcf.ZetaFn.apply(state["delta"], state["w"], plan, lo, hi)
        loss = (state["cot"] * zeta).sum()
        grad, = torch.autograd.grad(loss, state["delta"])
        return {"zeta": zeta.detach().float(), "grad": grad}
    if kind == "map_grouped":
        zeta, norm = plan.forward_grouped(state["delta"], state["w"], state["case"]["group"], state["range"])
    elif kind == "map_multi":
        zeta, norm = plan.forward_multi(state["fields"], state["range"])
    else:
        zeta, norm = plan.forward(state["delta"], state["w"], state.get("range"))
    return {"zeta": zeta.float(), "norm": norm.float()}


# ------------------------------------------------------------ what it must cost

def map_pairs(case):
    """Expected in-bin ordered pairs (mean pixel density, live pivots)."""
    npix = 12 * case["nside"] ** 2
    lo, hi = pivots_of(case, npix)
    live = 1.0 - math.sin(math.radians(20.0)) if case["w"] == "mask" else 1.0
    ann = (math.cos(math.radians(case["lo"])) - math.cos(math.radians(case["hi"]))) / 2.0
    return (hi - lo) * live / case.get("group", 1), npix * ann


def work(case):
    """Arithmetic: per in-bin pair a position angle and one complex multiply-add per multipole
    (24 + 10 m flops, twice that with the gradient); per pivot the contraction of its K(K+1)/2
    bin pairs per multipole.  Bytes: each map or point array read once, each output written once."""
    kind = case["kind"]
    if kind == "batch":
        parts = [work(c) for c in batch_members(case)]
        return {n: sum(p[n] for p in parts) for n in ("bytes", "flops")}
    k, m = case["k"], case["m"]
    out = 8.0 * (2 * (m + 1) * k * k + k * k)
    if kind.startswith("cat"):
        n = case["n"] + case["randoms"]
        ann = (math.cos(math.radians(case["lo"])) - math.cos(math.radians(case["hi"]))) / 2.0
        piv, nbr, size = n, n * ann, 32.0 * n
    else:
        piv, nbr = map_pairs(case)
        size = 8.0 * 12 * case["nside"] ** 2
    step = 2.0 if with_gradient(kind) else 1.0
    if kind == "map_multi":
        step, size = 3.0, 3.0 * size
    flops = step * piv * (nbr * (24 + 10 * m) + 4.0 * (m + 1) * k * (k + 1))
    return {"bytes": size + out + (0.5 * size if step == 2.0 else 0.0), "flops": flops}


# --------------------------------------------------- the estimator in 64 bits
#
# a_m^k(i) = sum_j w_j d_j exp(-i m phi_ij) over the points j of bin k about pivot i,
# W^k(i) = sum_j w_j; S = sum_i w_i d_i a^k1 conj(a^k2), D = sum_i w_i W^k1 W^k2, zeta = S / D.

EXACT_PAIRS = 4e9  # candidate pairs beyond which the 64-bit sums would take too long


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        got = [exact(c, seed * 1000 + i) for i, c in enumerate(batch_members(case))]
        z = [None if r is None else r["zeta"] for r in got]
        n = [None if r is None else r["norm"] for r in got]
        return {"zeta": z, "norm": n, "grad": [None if r is None else r["grad"] for r in got]}
    if kind.startswith("cat"):
        n = case["n"] + case["randoms"]
        if float(n) * n > 6e9:
            return None
        s = inputs(case, seed)
        return exact_sums(case, Catalogue(s["xyz"]), [(s["delta"], s["w"])], (0, n), s["cot"])
    piv, nbr = map_pairs(dict(case, lo=0.0, w="unit"))
    if piv * nbr * (3 if kind == "map_multi" else 1) > EXACT_PAIRS or 12 * case["nside"] ** 2 > 4e6:
        return None
    s = inputs(case, seed)
    fields = s.get("fields") or [(s["delta"], s["w"])]
    return exact_sums(case, Map(case["nside"], math.radians(case["hi"])), fields, pivots_of(case, 12 * case["nside"] ** 2),
                      s.get("cot"))


class Map:
    """Candidate neighbours of a block of pivots of one ring, with quarter squared chord and angle."""

    def __init__(self, nside, reach):
        self.z, self.s, self.n, self.shift, self.first = ring_table(nside)
        self.th, self.reach = np.arctan2(self.s, self.z), reach
        self.npoints = 12 * nside * nside

    def blocks(self, lo, hi, group):
        """(ring, pixel-in-ring of the geometry, caller's pixels [P, group] or -1)."""
        for i in range(len(self.n)):
            f, n = int(self.first[i]), int(self.n[i])
            if f >= hi or f + n <= lo:
                continue
            ng = -(-n // group)
            for a in range(0, ng, 2048):
                j = torch.arange(a, min(a + 2048, ng), device=DEV)
                mem = j[:, None] * group + torch.arange(group, device=DEV)[None, :]
                size = (mem < n).sum(1)
                mem = torch.where((mem < n) & (mem + f >= lo) & (mem + f < hi), mem + f, torch.full_like(mem, -1))
                keep = (mem >= 0).any(1)
                if bool(keep.any()):
                    yield i, (j * group + (size - 1) // 2)[keep], mem[keep]

    def near(self, i, q):
        """Yields (pixel [P, J], f [P, J], E, N) over blocks of rings; f = inf where there is no neighbour."""
        inside = np.nonzero(np.abs(self.th - self.th[i]) <= self.reach + 1e-9)[0]
        h2 = np.sin(0.5 * (self.th[inside] - self.th[i])) ** 2
        t = (math.sin(0.5 * self.reach) ** 2 - h2) / (self.s[inside] * self.s[i])
        half = np.where(t >= 1.0, self.n[inside] // 2,
                        self.n[inside] / math.pi * np.arcsin(np.sqrt(np.clip(t, 0.0, 1.0)))).astype(np.int64) + 2
        ph = math.pi * (2.0 * q.double() + float(self.shift[i])) / float(self.n[i])
        step = max(1, int(3e7) // int(q.numel() * (2 * half.max() + 1)))
        for a in range(0, len(inside), step):
            rs = inside[a:a + step]
            w = int(half[a:a + step].max())
            col = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(DEV)[None, :, None]  # noqa: E731
            n, s, sh, first = col(self.n[rs]), col(self.s[rs]), col(self.shift[rs]), col(self.first[rs])
            c = ph[:, None, None] * n / (2.0 * math.pi) - 0.5 * sh
            p = torch.round(c) + torch.arange(-w, w + 1, device=DEV, dtype=torch.float64)[None, None, :]
            o = p - c
            sp, cp = torch.sin(math.pi * o / n), torch.cos(math.pi * o / n)
            f = col(h2[a:a + step]) + float(self.s[i]) * s * sp * sp
            f = torch.where((o >= -0.5 * n) & (o < 0.5 * n), f, torch.full_like(f, math.inf))
            E = s * 2.0 * sp * cp
            N = col(np.sin(self.th[i] - self.th[rs])) + 2.0 * float(self.z[i]) * s * sp * sp
            yield tuple(v.flatten(1) for v in (p.long().remainder(n) + first, f, E, N))


class Catalogue:
    def __init__(self, xyz):
        self.x, self.npoints = xyz, xyz.shape[0]

    def blocks(self, lo, hi, group):
        step = max(1, int(2e7) // self.npoints)
        for a in range(lo, hi, step):
            j = torch.arange(a, min(a + step, hi), device=DEV)
            yield None, j, j[:, None]

    def near(self, i, q):
        p, x = self.x[q], self.x
        rho = torch.sqrt(p[:, 0] ** 2 + p[:, 1] ** 2)
        ex, ey = -p[:, 1] / rho, p[:, 0] / rho
        d = [x[None, :, c] - p[:, c:c + 1] for c in range(3)]
        f = 0.25 * (d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
        E = d[0] * ex[:, None] + d[1] * ey[:, None]
        N = d[0] * (-p[:, 2] * ey)[:, None] + d[1] * (p[:, 2] * ex)[:, None] + d[2] * rho[:, None]
        yield torch.arange(self.npoints, device=DEV)[None, :].expand(f.shape), f, E, N


def harmonics_of(E, N, m):
    """exp(-i j phi), j = 0..m, of the chosen pairs."""
    u = torch.complex(N, -E)
    u = u / u.abs()
    out, z = [], torch.ones_like(u)
    for j in range(m + 1):
        out.append(z)
        z = z * u
    return out


def pairs_of(geo, i, q, Ee, k):
    """The in-bin pairs of a block: (pivot in block, point, bin, E, N)."""
    for pix, f, E, N in geo.near(i, q):
        b = torch.bucketize(f, Ee, right=True) - 1  # E_k <= f < E_{k+1}
        row, col = torch.nonzero((b >= 0) & (b < k) & torch.isfinite(f), as_tuple=True)
        if row.numel():
            yield row, pix[row, col], b[row, col], E[row, col], N[row, col]


def exact_sums(case, geo, fields, span, cot):
    k, m, opt = case["k"], case["m"], case["opt"]
    Ee = torch.from_numpy(np.sin(0.5 * np.radians(edges_of(case))) ** 2).to(DEV)
    wd = [w.double() * d.double() for d, w in fields]
    w = [w.double() for _, w in fields]
    nf, group = len(fields), case.get("group", 1)
    S = torch.zeros(m + 1, k, k, dtype=torch.complex128, device=DEV)
    D = torch.zeros(k, k, dtype=torch.float64, device=DEV)

    def moments(i, q):
        P = q.numel()
        a = torch.zeros(nf, m + 1, P * k, dtype=torch.complex128, device=DEV)
        W = torch.zeros(nf, P * k, dtype=torch.float64, device=DEV)
        Q, QW = torch.zeros(P * k, dtype=torch.float64, device=DEV), torch.zeros(P * k, dtype=torch.float64, device=DEV)
        for row, pix, b, E, N in pairs_of(geo, i, q, Ee, k):
            at = row * k + b
            hs = harmonics_of(E, N, m)
            for f in range(nf):
                v = wd[f][pix]
                for j in range(m + 1):
                    x = torch.view_as_real(hs[j] * v)
                    torch.view_as_real(a[f, j]).index_add_(0, at, x)
                W[f].index_add_(0, at, w[f][pix])
            if opt == "subtract":
                Q.index_add_(0, at, wd[0][pix] ** 2)
                QW.index_add_(0, at, w[0][pix] ** 2)
        return a.view(nf, m + 1, P, k), W.view(nf, P, k), Q.view(P, k), QW.view(P, k)

    def pivot_sums(v, mem):
        return torch.where(mem >= 0, v[mem.clamp(min=0)], torch.zeros((), dtype=v.dtype, device=DEV)).sum(1)

    cycles = [(0, 0, 0)] if nf == 1 else [(0, 1, 2), (1, 2, 0), (2, 0, 1)]
    for i, q, mem in geo.blocks(*span, group):
        a, W, Q, QW = moments(i, q)
        if opt in ("bin_mean", "pivot_total"):
            by = W[0] if opt == "bin_mean" else W[0].sum(1, keepdim=True).expand(-1, k)
            inv = torch.where(by > 0, 1.0 / by, torch.zeros_like(by))
            a, W = a * inv, torch.ones_like(W)
        for p, x, y in cycles:
            c, cw = pivot_sums(wd[p], mem), pivot_sums(w[p], mem)
            S += torch.einsum("p,mpk,mpl->mkl", c.to(a.dtype), a[x], a[y].conj())
            D += torch.einsum("p,pk,pl->kl", cw, W[x], W[y])
            if opt == "subtract":
                S.diagonal(dim1=1, dim2=2).sub_((c[:, None] * Q).sum(0))
                D.diagonal().sub_((cw[:, None] * QW).sum(0))
    zeta = torch.where(D != 0, S / torch.where(D != 0, D, torch.ones_like(D)), torch.zeros_like(S))
    out = {"zeta": torch.view_as_real(zeta), "norm": D}
    if not with_gradient(case["kind"]):
        return out
    # dL/d(delta): the pivot's own term and both neighbour legs
    C = torch.where(D != 0, torch.complex(cot[..., 0], -cot[..., 1]) / torch.where(D != 0, D, torch.ones_like(D)),
                    torch.zeros_like(S))
    H = C + C.conj().transpose(1, 2)
    diag = torch.einsum("mkk->k", C).real
    grad = torch.zeros(geo.npoints, dtype=torch.float64, device=DEV)
    for i, q, mem in geo.blocks(*span, 1):
        a, W, Q, QW = moments(i, q)
        h = torch.einsum("mkl,mpl->mpk", H, a[0].conj())
        own = 0.5 * (a[0] * h).sum((0, 2)).real
        if opt == "subtract":
            own = own - (Q * diag).sum(1)
        pix0, c = mem[:, 0], wd[0][mem[:, 0]]
        grad.index_add_(0, pix0, w[0][pix0] * own)
        flat = h.reshape(m + 1, -1)
        for row, pix, b, E, N in pairs_of(geo, i, q, Ee, k):
            v = torch.zeros_like(E)
            for j, e in enumerate(harmonics_of(E, N, m)):
                v += (e * flat[j][row * k + b]).real
            if opt == "subtract":
                v -= 2.0 * diag[b] * wd[0][pix]
            grad.index_add_(0, pix, w[0][pix] * c[row] * v)
    out["grad"] = grad
    return {n: out[n] for n in ("zeta", "grad")} if case["kind"].endswith("_step") else out
