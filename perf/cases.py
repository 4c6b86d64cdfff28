"""What the speed of this framework is measured on.

A case is one call, or one fixed group of calls, of a user's Monte Carlo
program through the public classes:

  chain    one lattice that lives on the GPU is swept (Lattice.sweep), or swept
           and measured after every sweep (Lattice.sweep_measure), with the
           options such programs set (over-relaxation, the a0 sampler).
  analyse  a stored configuration, in device memory in the canonical FP64
           layout, is loaded and measured: plaquette, Polyakov loop, APE
           smearing, Wilson loops on the smeared links.
  batch    many independent lattices in one Batch: swept and then measured
           (Batch.sweep, plaquette, polyakov), or measured after every sweep
           (Batch.sweep_measure).

listed() holds the sizes of this framework's own configurations (8^4 FP64,
16^4, the 32^3 x 4 finite-temperature scan in FP32 and binary16, 64 uneven
lattices in a batch, 64^4) and others of the same ranges: a ragged lattice, a
large FP64 chain, and FP64 loops with an extent that is no power of two.
draw() spreads sizes, precisions and options over those ranges.

exact() is the same method in plain torch FP64, written from the definitions
in include/su2.h: Philox4x32-10 draws, the checkerboard heat bath, the
observables.  Links are held by parity (the layout of the link store), with
independent lattices of one shape stacked in front.
"""
import math

import numpy as np
import torch

from paper_1010_4834_gb300 import Batch, Lattice

MASK = 0xFFFFFFFF
SITES = 64 ** 4                      # the largest lattice measured
CHAIN_WORK = 8 * SITES               # FP32 site-sweeps of the largest chain
SLOW = {"f32": 1, "f16q": 1, "f64": 32}   # FP64 arithmetic runs at 1/64 of the FP32 rate
DTYPE = {"f64": torch.float64, "f32": torch.float32, "f16q": torch.float16}
LINK = {"f64": 32, "f32": 16, "f16q": 8}  # bytes of one stored link


def _links_too(case):
    """Whether a chain's links are among its outputs.  In 32-bit arithmetic a
    trial whose acceptance hangs on the last bit (about one in 2e7, more in
    Creutz's sampler) may go either way, and its link is then another one.
    Longer FP32 chains, and all in binary16, whose rounding widens that margin,
    are known by what they measure; over-relaxation, which spreads rounding,
    counts like length."""
    updates = 4 * math.prod(_dims(case["dims"])) * case["sweeps"]
    return case["prec"] == "f64" or (case["prec"] == "f32" and case["sampler"] == "kp" and not case["overrelax"]
                                     and case["sweeps"] <= 8 and updates <= 2200000)


def _chain(name, dims, prec, beta, sweeps, measure, overrelax=0, sampler="kp", tries=64):
    return {"name": name, "kind": "chain", "dims": dims, "prec": prec, "beta": beta, "sweeps": sweeps,
            "measure": measure, "overrelax": overrelax, "sampler": sampler, "tries": tries}


def _analyse(name, dims, prec, beta, steps, alpha, rmax, tmax):
    return {"name": name, "kind": "analyse", "dims": dims, "prec": prec, "beta": beta, "steps": steps,
            "alpha": alpha, "rmax": rmax, "tmax": tmax}


def _batch(name, shapes, prec, sweeps, measure):
    return {"name": name, "kind": "batch", "shapes": shapes, "prec": prec, "sweeps": sweeps, "measure": measure}


def listed():
    return [
        # the smallest chain a study starts with, at the reference precision
        _chain("chain_8^4_f64_measured", "8x8x8x8", "f64", 2.4, 16, True),
        # an ordinary zero-temperature chain, decorrelation sweeps between measurements
        _chain("chain_16^4_f32", "16x16x16x16", "f32", 2.5, 8, False),
        # one coupling of the finite-temperature scan, as its production runs are
        # made: over-relaxation before each heat-bath sweep
        _chain("chain_32^3x4_f32_or", "32x32x32x4", "f32", 2.3, 8, True, overrelax=1),
        # the same lattice with binary16 links
        _chain("chain_32^3x4_f16q", "32x32x32x4", "f16q", 2.3, 8, True),
        # uneven extents, no power of two; the paper's own sampler
        _chain("chain_ragged_f32_creutz", "20x12x18x10", "f32", 2.2, 8, True, sampler="creutz"),
        # a production-size chain at the reference precision
        _chain("chain_24^3x32_f64", "24x24x24x32", "f64", 2.5, 4, False),
        # the largest lattice: the benchmark's measured sweeps
        _chain("chain_64^4_f32_measured", "64x64x64x64", "f32", 2.6, 8, True),
        # static-potential measurements on a stored configuration, small and largest
        _analyse("analyse_16^4_f32", "16x16x16x16", "f32", 2.5, 25, 0.7, 8, 8),
        _analyse("analyse_64^4_f32", "64x64x64x64", "f32", 2.6, 25, 0.7, 16, 16),
        # the same at the reference precision, with a time extent of 24
        _analyse("analyse_20^3x24_f64", "20x20x20x24", "f64", 2.5, 10, 0.5, 10, 12),
        # 64 independent lattices of uneven sizes swept together, then measured
        _batch("batch_64_uneven_f32", "8x8x8x8*16,12x12x12x12*16,16x16x16x16*16,24x24x24x6*16", "f32", 8, False),
        # the whole finite-temperature scan as one batch, measured every sweep
        _batch("batch_scan_16x32^3x4_f32", "32x32x32x4*16", "f32", 8, True),
    ]


def _even(rng, lo, hi):
    """An even extent, its logarithm uniform."""
    return max(lo, min(hi, 2 * round(0.5 * math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def _extents(rng, lo, hi, most):
    """A lattice: spatial cubes with a time extent of their own, or four
    independent extents (one in three)."""
    while True:
        n = [_even(rng, lo, hi) for _ in range(4)]
        if rng.random() < 0.67:
            n[1] = n[2] = n[0]
        if 256 <= math.prod(n) <= most:
            return n


def draw(rng):
    kind = rng.choice(["chain"] * 6 + ["analyse"] * 3 + ["batch"] * 2)
    beta = round(rng.uniform(2.0, 2.8), 3)
    prec = rng.choice(["f32", "f32", "f32", "f16q", "f64"])
    if kind == "chain":
        n = _extents(rng, 4, 64, SITES // SLOW[prec] * (1 if prec != "f64" else 2))
        overrelax = rng.choice([0, 0, 0, 1, 1, 2]) if prec != "f16q" else 0
        most = CHAIN_WORK // (SLOW[prec] * math.prod(n) * (1 + overrelax))
        # rounding grows along a chain, most in over-relaxation: 8 of those at most
        sweeps = max(1, min(most, _even(rng, 2, 16 if prec == "f64" else 8), 8 // overrelax if overrelax else 16))
        sampler = rng.choice(["kp", "kp", "kp", "creutz"])
        return _chain_of(n, prec, beta, sweeps, rng.random() < 0.5, overrelax, sampler,
                         rng.choice([64, 64, 64, 1]))
    if kind == "analyse":
        n = _extents(rng, 4, 64, SITES // (16 if prec == "f64" else 1))
        rmax = rng.randint(1, min(16, *n[:3]))
        tmax = rng.randint(1, min(16, n[3]))
        c = _analyse("", "x".join(map(str, n)), prec, beta, rng.choice([0, 5, 10, 25]),
                     rng.choice([0.3, 0.5, 0.7]), rmax, tmax)
        del c["name"]
        return c
    shapes, sites, least = [], 0, SITES
    for _ in range(rng.randint(1, 4)):
        n = _extents(rng, 4, 32, 32 ** 3 * 4)
        count = rng.randint(1, 16)
        v = math.prod(n)
        # lattices whose sizes differ by more than the batch has multiprocessors
        # for are not batched together
        if sites + count * v <= min(1 << 21, 100 * min(least, v)):
            sites, least = sites + count * v, min(least, v)
            shapes.append("%s*%d" % ("x".join(map(str, n)), count))
    prec = rng.choice(["f32", "f32", "f16q", "f64"])
    c = _batch("", ",".join(shapes) or "8x8x8x8*3", prec, 2 if prec == "f64" else _even(rng, 2, 8), rng.random() < 0.5)
    del c["name"]
    return c


def _chain_of(n, *options):
    c = _chain("", "x".join(map(str, n)), *options)
    del c["name"]
    return c


def _dims(text):
    return tuple(int(t) for t in text.split("x"))


def _lattices(case):
    """(extents, beta) of every lattice of a case, in order."""
    if case["kind"] != "batch":
        return [(_dims(case["dims"]), case["beta"])]
    dims = [_dims(t.split("*")[0]) for t in case["shapes"].split(",") for _ in range(int(t.split("*")[1]))]
    return [(d, 2.0 + 0.8 * (i * 7 % len(dims) + 0.5) / len(dims)) for i, d in enumerate(dims)]


def _configuration(dims, beta, seed):
    """Links like those of a thermalised configuration at this coupling: a unit
    quaternion near 1 on every link, spread so that the mean plaquette is about
    the ensemble's, then a random gauge transformation.  Canonical layout
    (sites, direction, component), FP64, on the GPU."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    n = dims[::-1]
    mean = max(0.05, 1.0 - 0.75 / beta if beta > 2.2 else beta / 4 + 0.02 * beta ** 3)
    spread = math.sqrt((mean ** -0.5 - 1.0) / 3.0)

    def unit(q):
        return q.div_(q.square().sum(-1, keepdim=True).sqrt_())

    u = torch.randn(*n, 4, 4, generator=g, device="cuda", dtype=torch.float32).double().mul_(spread)
    u[..., 0] = 1.0
    unit(u)
    w = unit(torch.randn(*n, 4, generator=g, device="cuda", dtype=torch.float32).double())
    for mu in range(4):
        a = torch.stack(_mul(w.unbind(-1), u[..., mu, :].unbind(-1)), -1)
        b = w.roll(-1, 3 - mu)
        u[..., mu, :] = torch.stack(_mul_nd(a.unbind(-1), b.unbind(-1)), -1)
    unit(u)
    return u.reshape(-1, 4, 4)


def _start(case, seed):
    return [_configuration(d, b, seed * 4099 + i) for i, (d, b) in enumerate(_lattices(case))]


def prepare(case, seed):
    prec, start = case["prec"], _start(case, seed)
    if case["kind"] == "batch":
        every = _lattices(case)
        b = Batch([d for d, _ in every], [x for _, x in every], seed=seed, start="cold", prec=prec)
        for i, u in enumerate(start):
            b.set_links(i, u.cpu().numpy())
        b.tune()
        return {"case": case, "batch": b}
    dims = _dims(case["dims"])
    lat = Lattice(dims, case["beta"], seed=seed, start="cold", prec=prec)
    if case["kind"] == "analyse":
        torch.cuda.synchronize()
        return {"case": case, "lattice": lat, "links": start[0]}
    lat.set_options(case["tries"], case["sampler"])
    lat.set_overrelax(case["overrelax"])
    lat.set_links(start[0])
    # the store opens the lattice's device buffer: eight (direction, parity)
    # classes of V / 2 links
    store = lat._buf[:4 * lat.volume * LINK[prec]].view(DTYPE[prec]).view(8, lat.volume // 2, 4)
    return {"case": case, "lattice": lat, "store": store}


def run(state):
    case = state["case"]
    if case["kind"] == "chain":
        lat = state["lattice"]
        if case["measure"]:
            out = {"history": lat.sweep_measure(case["sweeps"])}
        else:
            lat.sweep(case["sweeps"])
            out = {} if _links_too(case) else {"means": np.append(lat.plaquette(), lat.polyakov())}
        if _links_too(case):
            out["links"] = state["store"]
        return out
    if case["kind"] == "analyse":
        lat = state["lattice"]
        lat.set_links(state["links"])
        out = {"means": np.append(lat.plaquette(), lat.polyakov())}
        lat.ape_smear(case["alpha"], case["steps"])
        out["wilson"] = lat.wilson_loops(case["rmax"], case["tmax"], smeared=True)
        return out
    b = state["batch"]
    if case["measure"]:
        return {"history": b.sweep_measure(case["sweeps"])}
    b.sweep(case["sweeps"])
    return {"means": np.column_stack([b.plaquette(), b.polyakov()])}


def work(case):
    """Every sweep (or smearing step) reads and writes each link it changes
    once; a measurement reads each link once.  A checkerboard schedule of eight
    substeps moves more: 3.5 + 0.5 of the 4 link classes a substep, so 4 times
    the sweep's bytes here.  Operations: 12 quaternion products of 28 a staple
    sum, 110 for the draw and the composition of a link."""
    link = LINK[case["prec"]]
    sites = sum(math.prod(d) for d, _ in _lattices(case))
    if case["kind"] == "analyse":
        loops = 3 * case["rmax"] * case["tmax"] * 8 + 3 * case["rmax"] * 28
        return {"bytes": sites * (4 * 32 + 4 * link + 3 * 2 * link * case["steps"] + 4 * link),
                "flops": sites * (6 * 63 + 28 + 3 * 140 * case["steps"] + loops)}
    sweeps = case["sweeps"]
    each = 1 + case.get("overrelax", 0)
    return {"bytes": sites * 4 * 2 * link * sweeps * each,
            "flops": sites * 4 * sweeps * (470 + 450 * (each - 1))}


def tolerance(case):
    """About four times the distance to exact() seen over listed and drawn
    cases.  Means of FP32 chains: an accept decision that rounding turns (one
    in 2e7) changes a handful of the N links and, through them, their
    neighbours in later sweeps (more with over-relaxation and in Creutz's
    sampler, and more in a batch, whose small lattices weigh as much as its
    large ones)."""
    prec = case["prec"]
    if case["kind"] == "analyse":
        return {"f64": {"rel": 2e-15}, "f32": {"rel": 6e-6}, "f16q": {"rel": 3e-5}}[prec]
    batch, relaxed = case["kind"] == "batch", case.get("overrelax", 0) > 0
    if prec == "f64":
        return {"rel": 4e-12, "max": 4e-10} if relaxed else {"rel": 4e-13, "max": 2e-11}
    if not batch and _links_too(case):
        return {"rel": 6e-6}
    links = 4 * sum(math.prod(d) for d, _ in _lattices(case))
    if prec == "f16q":
        return {"rel": min(0.03, 5e-5 + (10.0 if batch else 1.0) / math.sqrt(links))}
    flips = math.sqrt(2.0 + 1e-7 * links * case["sweeps"])
    spread = 1000.0 if batch or relaxed else 400.0 if case["sampler"] == "creutz" else 100.0
    return {"rel": min(0.03, 1e-6 + spread * flips / links)}


# -- the method in plain torch FP64 ----------------------------------------
# A quaternion field is a tuple of four tensors of shape (lattices, N3, N2,
# N1, N0/2): the sites of one parity.  U[mu][p] is direction mu on parity p.

def _mul(a, b):
    return (a[0] * b[0] - a[1] * b[1] - a[2] * b[2] - a[3] * b[3],
            a[0] * b[1] + a[1] * b[0] - a[2] * b[3] + a[3] * b[2],
            a[0] * b[2] + a[2] * b[0] - a[3] * b[1] + a[1] * b[3],
            a[0] * b[3] + a[3] * b[0] - a[1] * b[2] + a[2] * b[1])


def _dag(a):
    return (a[0], -a[1], -a[2], -a[3])


def _mul_nd(a, b):
    return _mul(a, _dag(b))


def _mul_dn(a, b):
    return _mul(_dag(a), b)


def _dot(a, b):
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2] + a[3] * b[3]


def _add(a, b):
    return tuple(x + y for x, y in zip(a, b))


def _scale(a, s):
    return tuple(x * s for x in a)


class _Checkerboard:
    def __init__(self, dims):
        self.dims = dims
        n0, n1, n2, n3 = dims
        t, z, y = torch.meshgrid(torch.arange(n3, device="cuda"), torch.arange(n2, device="cuda"),
                                 torch.arange(n1, device="cuda"), indexing="ij")
        row = (y + n1 * (z + n2 * t)).unsqueeze(-1)
        odd = ((t + z + y) & 1).unsqueeze(-1)
        half = torch.arange(n0 // 2, device="cuda")
        self.x0odd = [(odd ^ p).bool() for p in (0, 1)]            # x0 & 1 on parity p, by row
        self.site = [2 * half + (odd ^ p) + n0 * row for p in (0, 1)]

    def shift(self, q, p, mu, step):
        """The field q, given on the parity other than p, at x + step mu for the sites x of parity p."""
        if mu:
            return tuple(c.roll(-step, 4 - mu) for c in q)
        odd = self.x0odd[p] if step > 0 else ~self.x0odd[p]
        return tuple(torch.where(odd, c.roll(-step, 4), c) for c in q)

    def split(self, full):
        """Canonical links (lattices, sites, 4, 4) to U[mu][p]."""
        full = full.reshape(full.shape[0], -1, 4, 4)
        return [[tuple(full[:, self.site[p].reshape(-1), mu, c].reshape(full.shape[0], *self.site[p].shape)
                       for c in range(4)) for p in (0, 1)] for mu in range(4)]

    def staple(self, U, mu, p, directions=range(4)):
        """U_nu(x) U_mu(x+nu) U_nu(x+mu)^+ + U_nu(x-nu)^+ U_mu(x-nu) U_nu(x-nu+mu), summed over nu != mu."""
        s = None
        for nu in directions:
            if nu == mu:
                continue
            up = _mul_nd(_mul(U[nu][p], self.shift(U[mu][1 - p], p, nu, 1)), self.shift(U[nu][1 - p], p, mu, 1))
            # the backward term, formed at x - nu (parity 1 - p) and brought to x
            down = _mul(_mul_dn(U[nu][1 - p], U[mu][1 - p]), self.shift(U[nu][p], 1 - p, mu, 1))
            up = _add(up, self.shift(down, p, nu, -1))
            s = up if s is None else _add(s, up)
        return s

    def plaquette(self, U):
        """All, spatial, space-time means, a row for each lattice."""
        space = time = 0.0
        for p in (0, 1):
            for mu in range(4):
                for nu in range(mu + 1, 4):
                    a = _mul(U[mu][p], self.shift(U[nu][1 - p], p, mu, 1))
                    b = _mul(U[nu][p], self.shift(U[mu][1 - p], p, nu, 1))
                    v = _dot(a, b).sum((1, 2, 3, 4))
                    space, time = (space, time + v) if nu == 3 else (space + v, time)
        n = 3.0 * math.prod(self.dims)
        return torch.stack([(space + time) / (2 * n), space / n, time / n], -1)

    def polyakov(self, U):
        total = 0.0
        for p in (0, 1):
            q = None
            for t in range(self.dims[3]):
                u = tuple(c[:, t] for c in U[3][p ^ (t & 1)])
                q = u if q is None else _mul(q, u)
            total = total + q[0].sum((1, 2, 3))
        return total / math.prod(self.dims[:3])


def _philox(site, tag, sweep, draw, seed):
    """Philox4x32-10, the counter words in int64 tensors below 2^32."""
    def halves(m, c):
        high = (m * (c >> 16) + ((m * (c & 0xFFFF)) >> 16)) >> 16
        return high, (m * c) & MASK

    x, y, z, w = site, tag, torch.full_like(site, sweep), torch.full_like(site, draw)
    k0, k1 = seed & MASK, (seed >> 32) & MASK
    for _ in range(10):
        h0, l0 = halves(0xD2511F53, x)
        h1, l1 = halves(0xCD9E8D57, z)
        x, y, z, w = h1 ^ y ^ k0, l1, h0 ^ w ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & MASK, (k1 + 0xBB67AE85) & MASK
    return x, y, z, w


def _uniform(x, prec):
    return (x.double() + 0.5) * 2.0 ** -32 if prec == "f64" else ((x >> 9).double() + 0.5) * 2.0 ** -23


def _direction(words, first, prec):
    """cos(theta) and phi of the new link's direction: from draw 0 in FP64, from
    the low bits of the accepting trial's words otherwise."""
    if prec == "f64":
        return 2.0 * _uniform(first[0], prec) - 1.0, 2.0 * math.pi * _uniform(first[1], prec)
    c = ((words[0] & 511) << 9) | (words[1] & 511)
    f = ((words[2] & 511) << 9) | (words[3] & 511)
    return (2 * c + 1).double() * 2.0 ** -18 - 1.0, 2.0 * math.pi * (f.double() + 0.5) * 2.0 ** -18


def _heat_bath(board, U, mu, p, beta, lattice, sweep, seed, case):
    """One substep.  beta and lattice: one value for each stacked lattice."""
    prec, tries = case["prec"], case.get("tries", 64)
    creutz = case.get("sampler", "kp") == "creutz"
    s = board.staple(U, mu, p)
    k = _dot(s, s).sqrt()
    w = _scale(s, 1.0 / k)
    shape = (-1, 1, 1, 1, 1)
    alpha = beta.view(shape) * k
    site = board.site[p].expand(k.shape)
    tag = (mu | (lattice.view(shape) << 2)).expand(k.shape)
    old = U[mu][p]
    left = torch.arange(k.numel(), device="cuda")
    new = [c.reshape(-1).clone() for c in old]
    site, tag, alpha = site.reshape(-1), tag.reshape(-1), alpha.reshape(-1)
    w = [c.reshape(-1) for c in w]
    for trial in range(1, tries + 1):
        st, tg, al = site[left], tag[left], alpha[left]
        words = _philox(st, tg, sweep, trial, seed)
        u = [_uniform(x, prec) for x in words]
        if creutz:
            e = torch.exp(-2.0 * al)
            a0 = 1.0 + torch.log(e + (1.0 - e) * u[0]) / al
            good = u[1] * u[1] <= 1.0 - a0 * a0
        else:
            delta = -(u[0].log() + torch.cos(2.0 * math.pi * u[1]).square() * u[2].log()) / (2.0 * al)
            a0 = 1.0 - 2.0 * delta
            good = u[3] * u[3] <= 1.0 - delta
        at = good.nonzero().squeeze(-1)
        link = left[at]
        first = _philox(st[at], tg[at], sweep, 0, seed) if prec == "f64" else None
        cos_t, phi = _direction([x[at] for x in words], first, prec)
        a0 = a0[at]
        sin_t = (1.0 - cos_t * cos_t).clamp_min(0).sqrt()
        rad = (1.0 - a0 * a0).clamp_min(0).sqrt()
        q = _mul((a0, rad * sin_t * phi.cos(), rad * sin_t * phi.sin(), rad * cos_t), [c[link] for c in w])
        for c in range(4):
            new[c][link] = q[c]
        left = left[(~good).nonzero().squeeze(-1)]
        if not left.numel():
            break
    U[mu][p] = tuple(n.view_as(o) for n, o in zip(new, old))


def _overrelax(board, U, mu, p, prec):
    s = board.staple(U, mu, p)
    w = _scale(s, 1.0 / _dot(s, s).sqrt())
    q = _mul(_mul_nd(w, U[mu][p]), w)
    U[mu][p] = q if prec == "f64" else _scale(q, 1.0 / _dot(q, q).sqrt())


def _stored(u, prec):
    """Links as the store of this precision holds them, for the arithmetic."""
    if prec == "f16q":
        u = u.half().double()
        return u / u.square().sum(-1, keepdim=True).sqrt()
    return u.float().double() if prec == "f32" else u


def _sweeps(case, dims, start, beta, lattice, seed):
    """The chain of stacked lattices: (U, a list of history rows)."""
    board = _Checkerboard(dims)
    U = board.split(_stored(start, case["prec"]))
    rows = []
    for sweep in range(case["sweeps"]):
        for _ in range(case.get("overrelax", 0)):
            for mu in range(4):
                for p in (0, 1):
                    _overrelax(board, U, mu, p, case["prec"])
        for mu in range(4):
            for p in (0, 1):
                _heat_bath(board, U, mu, p, beta, lattice, sweep, seed, case)
        if case["measure"] or sweep == case["sweeps"] - 1:
            rows.append(torch.cat([board.plaquette(U), board.polyakov(U).unsqueeze(-1)], -1))
    return U, torch.stack(rows)


def _smear(U, board, steps, alpha):
    for _ in range(steps):
        new = []
        for mu in range(3):
            new.append([])
            for p in (0, 1):
                s = board.staple(U, mu, p, range(3))
                q = _add(_scale(U[mu][p], 1.0 - alpha), _scale(s, 0.25 * alpha))
                new[mu].append(_scale(q, 1.0 / _dot(q, q).sqrt()))
        U = new + [U[3]]
    return U


def _wilson(board, smeared, links, rmax, tmax):
    """W(R, T) multiplied out, on full fields (N3, N2, N1, N0)."""
    n0, n1, n2, n3 = board.dims

    def full(halves):
        out = []
        for c in range(4):
            f = torch.empty(n3 * n2 * n1 * n0, device="cuda", dtype=torch.float64)
            for p in (0, 1):
                f[board.site[p].reshape(-1)] = halves[p][c].reshape(-1)
            out.append(f.view(n3, n2, n1, n0))
        return tuple(out)

    def at(q, step, axis):
        return tuple(c.roll(-step, axis) for c in q)

    time = full(links[3])
    out = torch.zeros(rmax, tmax, device="cuda", dtype=torch.float64)
    for mu in range(3):
        u = full(smeared[mu])
        lines = [u]
        for r in range(1, rmax):
            lines.append(_mul(lines[-1], at(u, r, 3 - mu)))
        column = time
        for t in range(1, tmax + 1):
            if t > 1:
                column = _mul(column, at(time, t - 1, 0))
            for r in range(1, rmax + 1):
                a = _mul(lines[r - 1], at(column, r, 3 - mu))
                b = _mul(column, at(lines[r - 1], t, 0))
                out[r - 1, t - 1] += _dot(a, b).mean() / 3.0
    return out


def exact(case, seed):
    every, start = _lattices(case), _start(case, seed)
    if case["kind"] == "analyse":
        board = _Checkerboard(every[0][0])
        U = board.split(_stored(start[0], case["prec"]).unsqueeze(0))
        S = _smear(U, board, case["steps"], case["alpha"])
        return {"means": torch.cat([board.plaquette(U)[0], board.polyakov(U)]),
                "wilson": _wilson(board, S, U, case["rmax"], case["tmax"])}
    groups = {}
    for i, (d, _) in enumerate(every):
        groups.setdefault(d, []).append(i)
    rows = [None] * len(every)
    for d, members in groups.items():
        beta = torch.tensor([every[i][1] for i in members], device="cuda", dtype=torch.float64)
        lattice = torch.tensor(members, device="cuda")
        U, h = _sweeps(case, d, torch.stack([start[i] for i in members]), beta, lattice, seed)
        for k, i in enumerate(members):
            rows[i] = h[:, k]
    if case["kind"] == "batch":
        h = torch.stack(rows, 1)
        return {"history": h} if case["measure"] else {"means": h[-1]}
    out = {"history": rows[0]} if case["measure"] else {} if _links_too(case) else {"means": rows[0][-1]}
    if _links_too(case):
        out["links"] = torch.stack([torch.stack([c.reshape(-1) for c in U[mu][p]], -1)
                                    for mu in range(4) for p in (0, 1)])
    return out
