"""The work a user of this library has it do, as measurable cases.

A case is a dict of plain values; its "kind" names the call sequence:

  bin        count maps of two nested boxes (Sec. 2.4; ufc_bin)
  periodic   count maps of one box with its periodic images (ufc_bin)
  snapshots  count maps of a snapshot-mode lightcone (ufc_bin_snapshots)
  map        one whole realisation: bin, kappa map with moments and PDF,
             statistics vector, covariance update
  kappa      kappa map, moments and PDF of given count maps
  adjoint    gradients of the map's statistics (fused with the map, or alone)
  spectrum   a_lm, C_l and band powers of a map
  smooth     beam, synthesis and statistics of the smoothed map
  batch      statistics and covariance of many realisations in one call

Sizes follow the package's workloads (two nested boxes of 2000 and 6400
Mpc/h, 40 shells at Nside 512 or 60 at Nside 1024, 150 realisations), the
benchmark's legs and the tests; draw() spreads over the ranges between the
smallest and the largest of them.
"""
import math

import numpy as np
import torch

from paper_1801_05745_gb300 import api, synth

DEV = "cuda"
Z_LO, Z_HI = 0.1, 1.5           # redshift range of the nested lightcone
L1, L2, R_SWITCH = 2000.0, 6400.0, 1000.0
SIG1, SIG2 = 5.0, 20.0          # blob sizes of the synthetic particles
NBINS = 200
ARCMIN = math.pi / (180.0 * 60.0)


def listed():
    return [
        # The periodic 500 Mpc/h box with four image layers: the smallest
        # binning workload, every image of few particles.
        {"name": "bin-periodic-64", "kind": "periodic", "nside": 64, "nshell": 10, "n": 64 ** 3,
         "layers": 4},
        # One small realisation of a covariance run, map at a time: short
        # kernels, so launches and host work count.
        {"name": "map-small-64", "kind": "map", "nside": 64, "nshell": 40, "n1": 262144,
         "n2": 262147},
        # The nested lightcone at the size of one covariance realisation.
        {"name": "bin-nested-512", "kind": "bin", "nside": 512, "nshell": 40, "n1": 512 ** 3,
         "n2": 512 ** 3},
        # The full-size map of the benchmark.
        {"name": "bin-full-1024", "kind": "bin", "nside": 1024, "nshell": 60, "n1": 1024 ** 3,
         "n2": 1024 ** 3},
        # Snapshot outputs every second shell, each a whole box read for two
        # shells only; a count that no tile divides.
        {"name": "snapshots-512", "kind": "snapshots", "nside": 512, "nshell": 30, "nsnap": 15,
         "n": 200 ** 3 + 1},
        # The full-size map from its counts.
        {"name": "kappa-full-1024", "kind": "kappa", "nside": 1024, "nshell": 60},
        # Map and gradient in one call, as a training or fitting step has it.
        {"name": "adjoint-full-1024", "kind": "adjoint", "nside": 1024, "nshell": 60,
         "fused": True, "with_g": False},
        # The paper's own 140 shells; gradient alone, with a cotangent of the
        # map itself (what the autograd function's backward calls).
        {"name": "adjoint-140-512", "kind": "adjoint", "nside": 512, "nshell": 140,
         "fused": False, "with_g": True},
        # The full-sky C_l of the full-size map, and of a small one with an
        # lmax that no tile divides.
        {"name": "spectrum-1024", "kind": "spectrum", "nside": 1024, "lmax": 3071},
        {"name": "spectrum-64", "kind": "spectrum", "nside": 64, "lmax": 150},
        # One smoothing scale (10.8 arcmin) of an Nside-512 map.
        {"name": "smooth-512", "kind": "smooth", "nside": 512, "lmax": 1535, "arcmin": 10.8},
        # 150 small realisations of Poisson-varied size in one call.
        {"name": "batch-150-64", "kind": "batch", "nside": 64, "nshell": 40, "nreal": 150,
         "n": 64 ** 3},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _pow2(rng, lo, hi):
    return 1 << rng.randint(lo.bit_length() - 1, hi.bit_length() - 1)


def draw(rng):
    kind = rng.choice(["bin", "periodic", "snapshots", "map", "kappa", "adjoint", "spectrum",
                       "smooth", "batch"])
    c = {"kind": kind}
    if kind == "bin":
        # at least one particle per few pixels, as real lightcones have
        c.update(nside=_pow2(rng, 64, 1024), nshell=rng.randint(10, 60))
        lo = 12 * c["nside"] ** 2
        c.update(n1=_log(rng, lo, 64 * lo), n2=_log(rng, lo, 64 * lo))
    elif kind == "periodic":
        c.update(nside=_pow2(rng, 32, 256), nshell=rng.randint(4, 20), n=_log(rng, 5000, 400000),
                 layers=rng.randint(1, 4))
    elif kind == "snapshots":
        c.update(nside=_pow2(rng, 128, 1024), nsnap=rng.randint(3, 30), n=_log(rng, 3e5, 3e7))
        c.update(nshell=c["nsnap"] * rng.randint(1, 2))
    elif kind == "map":
        c.update(nside=_pow2(rng, 16, 256), nshell=rng.randint(4, 60), n1=_log(rng, 2e4, 4e6),
                 n2=_log(rng, 2e4, 4e6))
    elif kind == "kappa":
        c.update(nside=_pow2(rng, 32, 1024), nshell=rng.randint(4, 140))
    elif kind == "adjoint":
        c.update(nside=_pow2(rng, 32, 1024), nshell=rng.randint(4, 140), fused=rng.random() < 0.5,
                 with_g=rng.random() < 0.5)
    elif kind == "spectrum":
        c.update(nside=_pow2(rng, 32, 1024))
        c.update(lmax=rng.randint(c["nside"], 3 * c["nside"] - 1))
    elif kind == "smooth":
        c.update(nside=_pow2(rng, 32, 1024))
        c.update(lmax=rng.randint(c["nside"], 3 * c["nside"] - 1),
                 arcmin=round(rng.uniform(2.0, 60.0), 1))
    else:
        c.update(nside=_pow2(rng, 16, 64), nshell=rng.randint(8, 40), nreal=rng.randint(8, 200),
                 n=_log(rng, 1e4, 3e5))
    return c


# ---- set-up shared by the kinds ---------------------------------------------------
def _cosmo():
    return api.make_cosmo(0.3, 0.7, 1)


def _source():
    return api.make_source(kind=1, alpha=2.0, beta=1.5, z0=0.5, z_max=1.5)


def _nested(nshell, n1, n2):
    """(z edges, chi edges, boxes) of the two nested boxes."""
    z = np.linspace(Z_LO, Z_HI, nshell + 1)
    chi = api.chi_edges(_cosmo(), z)
    split = int(np.argmin(np.abs(chi - R_SWITCH)))
    boxes = [api.make_box(L1, [L1 / 2] * 3, n1, 0, split),
             api.make_box(L2, [L2 / 2] * 3, n2, split, nshell)]
    return z, chi, boxes


def _density(chi, boxes, npix):
    """Mean particles per pixel of every shell."""
    vol = 4.0 / 3.0 * math.pi * (chi[1:] ** 3 - chi[:-1] ** 3)
    return np.array([v * next(b.n_total / b.L ** 3 for b in boxes if b.shell_lo <= i < b.shell_hi)
                     / npix for i, v in enumerate(vol)])


def _range(A, C, dens, spread=0.0):
    """A PDF range of +- 6 sigma around the expected mean of the map."""
    mean = float((A * dens).sum() - C)
    sig = math.sqrt(float((A * A * dens * (1.0 + dens * spread)).sum()))
    return mean - 6 * sig, mean + 6 * sig


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _counts(dens, npix, seed):
    """Poisson counts around a lognormal density field."""
    g = _gen(seed)
    out = torch.empty((len(dens), npix), dtype=torch.int32, device=DEV)
    for b, d in enumerate(dens):
        f = torch.randn(npix, generator=g, device=DEV)
        rate = torch.exp(0.5 * f - 0.125).mul_(float(d))
        out[b] = torch.poisson(rate, generator=g).to(torch.int32)
    return out


def _map(npix, seed):
    """A convergence-like map: noise with a skewed tail."""
    g = _gen(seed)
    a = torch.randn(npix, generator=g, device=DEV)
    b = torch.randn(npix, generator=g, device=DEV)
    return (0.01 * a + 0.004 * (b * b - 1.0)).contiguous()


def _coeffs(s, derivs=False):
    return api.kappa_coeffs(_cosmo(), s["boxes"], s["z"], s["nside"], _source(), derivs=derivs)


def prepare(case, seed):
    k = case["kind"]
    s = {"kind": k, "ctx": api.context(0), "nside": case["nside"]}
    npix = 12 * case["nside"] ** 2
    if k == "periodic":
        n, S = case["n"], case["nshell"]
        lo, hi = api.chi_edges(_cosmo(), [0.1, 0.5])
        s["chi"] = np.linspace(lo, hi, S + 1)
        s["boxes"] = [api.make_box(500.0, [250.0] * 3, n, 0, S, case["layers"])]
        s["xyz"] = [synth.particles_torch(n, 500.0, 5.0, seed, device=DEV)]
        s["counts"] = torch.empty((S, npix), dtype=torch.int32, device=DEV)
    elif k in ("bin", "map"):
        S = case["nshell"]
        s["z"], s["chi"], s["boxes"] = _nested(S, case["n1"], case["n2"])
        s["xyz"] = [synth.particles_torch(case["n1"], L1, SIG1, 2 * seed, device=DEV),
                    synth.particles_torch(case["n2"], L2, SIG2, 2 * seed + 1, device=DEV)]
        s["counts"] = torch.empty((S, npix), dtype=torch.int32, device=DEV)
        if k == "map":
            s["A"], _, s["C"] = _coeffs(s)
            s["range"] = _range(s["A"], s["C"], _density(s["chi"], s["boxes"], npix), 0.3)
            s["kappa"] = torch.empty(npix, dtype=torch.float32, device=DEV)
    elif k == "snapshots":
        S, m = case["nshell"], case["nsnap"]
        z = np.linspace(Z_LO, Z_HI, S + 1)
        s["chi"] = api.chi_edges(_cosmo(), z)
        s["of_shell"] = api.snapshot_assign(z, z[:-1:S // m])
        s["boxes"] = [api.make_box(L2, [L2 / 2] * 3, case["n"], 0, 1) for _ in range(m)]
        s["xyz"] = [synth.particles_torch(case["n"], L2, SIG2, 64 * seed + i, device=DEV)
                    for i in range(m)]
        s["counts"] = torch.empty((S, npix), dtype=torch.int32, device=DEV)
    elif k in ("kappa", "adjoint"):
        n = case["nside"] ** 3              # 512^3 at Nside 512, 1024^3 at Nside 1024
        s["z"], s["chi"], s["boxes"] = _nested(case["nshell"], n, n)
        dens = _density(s["chi"], s["boxes"], npix)
        s["A"], _, s["C"], s["dA"], s["dC"] = _coeffs(s, derivs=True)
        s["range"] = _range(s["A"], s["C"], dens, 0.3)
        s["counts"] = _counts(dens, npix, seed)
        s["kappa"] = torch.empty(npix, dtype=torch.float32, device=DEV)
        if k == "adjoint":
            s["fused"] = case["fused"]
            # the cotangent a loss on the map sends back: small, of either sign
            s["g"] = (torch.randn(npix, generator=_gen(seed + 1), device=DEV) / npix
                      if case["with_g"] else None)
    elif k == "spectrum":
        s["lmax"] = case["lmax"]
        s["map"] = _map(npix, seed)
    elif k == "smooth":
        lmax = s["lmax"] = case["lmax"]
        s["sigma"] = case["arcmin"] * ARCMIN
        # white-noise-like coefficients with a falling spectrum, a_l0 real
        nalm = (lmax + 1) * (lmax + 2) // 2
        re = torch.randn(nalm, generator=_gen(2 * seed), dtype=torch.float64, device=DEV)
        im = torch.randn(nalm, generator=_gen(2 * seed + 1), dtype=torch.float64, device=DEV)
        im[:lmax + 1] = 0.0
        l = _degrees(lmax).to(torch.float64)
        s["alm"] = torch.complex(re, im) * (1e-4 / (1.0 + l / 200.0))
        s["range"] = _smooth_range(lmax, s["sigma"])
    else:
        assert k == "batch"
        S, R, n = case["nshell"], case["nreal"], case["n"]
        rng = np.random.default_rng(seed)
        cap = int(1.5 * n + 6 * math.sqrt(1.5 * n)) + 8
        bufs = [[synth.particles_torch(cap, L, sg, 16 * seed + 2 * i + b, device=DEV)
                 for b, (L, sg) in enumerate(((L1, SIG1), (L2, SIG2)))] for i in range(8)]
        s["xyz"], s["boxes"], A, C = [], [], [], []
        for r in range(R):
            ns = [min(int(rng.poisson(rng.uniform(0.5, 1.5) * n)), cap) for _ in range(2)]
            at = [4 * int(rng.integers(0, (cap - m) // 4 + 1)) for m in ns]
            s["z"], s["chi"], boxes = _nested(S, max(1, ns[0]), max(1, ns[1]))
            s["xyz"].append([bufs[r % 8][b][at[b]:at[b] + ns[b]] for b in range(2)])
            s["boxes"].append(boxes)
            a, _, c = api.kappa_coeffs(_cosmo(), boxes, s["z"], case["nside"], _source())
            A.append(a)
            C.append(c)
        s["A"], s["C"] = np.array(A), np.array(C)
        s["range"] = _range(A[0], C[0], _density(s["chi"], s["boxes"][0], npix), 0.3)
        s["counts"] = torch.empty((S, npix), dtype=torch.int32, device=DEV)
        s["kappa"] = torch.empty(npix, dtype=torch.float32, device=DEV)
    return s


def run(s):
    k, ctx, nside = s["kind"], s["ctx"], s["nside"]
    if k in ("bin", "periodic"):
        return ctx.bin(s["xyz"], s["boxes"], s["chi"], nside, counts=s["counts"])
    if k == "snapshots":
        return ctx.bin_snapshots(s["xyz"], s["boxes"], s["of_shell"], s["chi"], nside,
                                 counts=s["counts"])
    if k == "map":
        state = api.welford_state(6 + NBINS, DEV)
        ctx.bin(s["xyz"], s["boxes"], s["chi"], nside, counts=s["counts"])
        kap, mom, pdf = ctx.kappa_stats(s["counts"], s["A"], s["C"], *s["range"], NBINS,
                                        kappa=s["kappa"])
        vec = ctx.stats_vector(mom, pdf)
        ctx.welford_update(vec.view(1, -1), state)
        return {"counts": s["counts"], "kappa": kap, "moments": mom, "pdf": pdf, "vector": vec,
                "state": state}
    if k == "kappa":
        kap, mom, pdf = ctx.kappa_stats(s["counts"], s["A"], s["C"], *s["range"], NBINS,
                                        kappa=s["kappa"])
        return {"kappa": kap, "moments": mom, "pdf": pdf}
    if k == "adjoint":
        # H is the sum of a cotangent whose variance and skewness parts sum to
        # zero: rounding alone without g, so it is left out of the results
        if s["fused"]:
            kap, mom, pdf, grad, G, H = ctx.kappa_stats_backward(
                s["counts"], s["A"], s["C"], s["dA"], s["dC"], *s["range"], NBINS, 1.0, 1.0,
                g_kappa=s["g"], kappa=s["kappa"])
            return {"kappa": kap, "moments": mom, "pdf": pdf, "grad": grad, "G": G}
        grad, G, H = ctx.kappa_backward(s["counts"], s["A"], s["C"], s["dA"], s["dC"], 1.0, 1.0,
                                        s["g"])
        return {"grad": grad, "G": G}
    if k == "spectrum":
        lmax = s["lmax"]
        alm = ctx.map2alm(s["map"], nside, lmax)
        cl = ctx.alm2cl(alm, lmax)
        band = ctx.cl_bin(cl, lmax, 10, 10, (lmax + 1 - 10) // 10)
        return {"alm": alm, "cl": cl, "band": band}
    if k == "smooth":
        sm = ctx.alm2map(ctx.alm_beam(s["alm"], s["lmax"], s["sigma"]), nside, s["lmax"])
        mom, pdf = ctx.map_stats(sm, nside, *s["range"], NBINS)
        return {"map": sm, "moments": mom, "pdf": pdf}
    state = api.welford_state(6 + NBINS, DEV)
    mom, pdf, vec = ctx.batched_stats(s["xyz"], s["boxes"], s["chi"], nside, s["A"], s["C"],
                                      *s["range"], NBINS, state, counts=s["counts"],
                                      kappa=s["kappa"])
    return {"moments": mom, "pdf": pdf, "vectors": vec, "state": state}


def _in_shells(case):
    """Expected particle images inside the shells of a binning case."""
    if case["kind"] == "periodic":
        lo, hi = map(float, api.chi_edges(_cosmo(), [0.1, 0.5]))
        reach = 500.0 * (case["layers"] + 0.5)
        hi, lo = min(hi, reach), min(lo, reach)
        return case["n"] * 4.0 / 3.0 * math.pi * (hi ** 3 - lo ** 3) / 500.0 ** 3
    z = np.array([Z_LO, Z_HI])
    lo, hi = map(float, api.chi_edges(_cosmo(), z))
    hi2 = min(hi, 0.62 * L2)                      # a sphere of the outer box's volume
    ball = lambda r: 4.0 / 3.0 * math.pi * r ** 3
    if case["kind"] == "snapshots":
        return case["n"] * (ball(hi2) - ball(lo)) / L2 ** 3
    n1, n2 = (case["n1"], case["n2"]) if "n1" in case else (case["n"], case["n"])
    return (n1 * (ball(R_SWITCH) - ball(lo)) / L1 ** 3 +
            n2 * (ball(hi2) - ball(R_SWITCH)) / L2 ** 3)


def work(case):
    """Inputs read once and outputs written once.  Arithmetic: per particle
    the squared distance and a comparison (10), per particle inside the
    shells its pixel (60); per pixel and shell a multiply-add, and for
    gradients three more; per (l, m, ring pair) the recurrence and the
    complex accumulation (8); per ring of n pixels 5 n log2 n."""
    k = case["kind"]
    npix = 12 * case["nside"] ** 2
    if k in ("bin", "periodic", "map"):
        n = case["n"] if k == "periodic" else case["n1"] + case["n2"]
        cells = case["nshell"] * npix
        b, f = 12 * n + 4 * cells, 10 * n + 60 * _in_shells(case)
        if k == "map":
            b += 4 * cells + 4 * npix
            f += 2 * cells + 10 * npix
        return {"bytes": b, "flops": f}
    if k == "snapshots":
        n = case["n"] * case["nsnap"]
        return {"bytes": 12 * n + 4 * case["nshell"] * npix, "flops": 10 * n + 60 * _in_shells(case)}
    if k == "kappa":
        cells = case["nshell"] * npix
        return {"bytes": 4 * cells + 4 * npix, "flops": 2 * cells + 10 * npix}
    if k == "adjoint":
        cells = case["nshell"] * npix
        maps = int(case["fused"]) + int(case["with_g"])
        return {"bytes": 4 * cells + 4 * npix * maps, "flops": 8 * cells + 20 * npix}
    if k in ("spectrum", "smooth"):
        lmax = case["lmax"]
        nalm = (lmax + 1) * (lmax + 2) // 2
        return {"bytes": 4 * npix + 16 * nalm,
                "flops": 8 * nalm * 2 * case["nside"] + 5 * npix * math.log2(4 * case["nside"])}
    n, R = 2 * case["n"] * case["nreal"], case["nreal"]
    return {"bytes": 12 * n + 8 * R * (16 + 2 * (6 + NBINS)) + 8 * (7 + NBINS) ** 2,
            "flops": 10 * n + 60 * R * _in_shells(case) + 2 * R * case["nshell"] * npix
            + 2 * R * (6 + NBINS) ** 2}


# ---- the same results in 64 bits ---------------------------------------------------
def _degrees(lmax):
    """l of every coefficient, m-major."""
    return torch.cat([torch.arange(m, lmax + 1, device=DEV) for m in range(lmax + 1)])


def _smooth_range(lmax, sigma):
    """+- 5 r.m.s. of a field with the spectrum of prepare()'s coefficients."""
    l = np.arange(lmax + 1)
    c = 1e-8 / (1.0 + l / 200.0) ** 2 * np.exp(-l * (l + 1.0) * sigma ** 2)
    sd = math.sqrt(float(((1 + 4 * l) * c).sum() / (4 * math.pi)))
    return -5 * sd, 5 * sd


def _moments(x):
    """The ten moments of a map of FP32 values held in FP64."""
    N = float(x.numel())
    mean = x.mean()
    d = x - mean
    m2, m3, m4 = (d ** 2).mean(), (d ** 3).mean(), (d ** 4).mean()
    vs = (N - 1) ** 2 / N ** 3 * m4 - (N - 1) * (N - 3) / N ** 3 * m2 * m2
    one = torch.ones((), dtype=torch.float64, device=x.device)
    return torch.stack([mean, m2, m3, m4, m3 / m2 ** 1.5, m4 / m2 ** 2 - 3.0, (N - 1) * m2 / N,
                        vs, m2 / vs, N * one])


def _histogram(x, lo, hi):
    b = torch.floor((x - lo) * (NBINS / (hi - lo))).long().clamp_(0, NBINS - 1)
    return torch.bincount(b[(x >= lo) & (x < hi)], minlength=NBINS)


def _kappa(counts, A, C):
    e = torch.zeros(counts.shape[1], dtype=torch.float64, device=counts.device)
    for b in range(counts.shape[0]):
        e += float(A[b]) * counts[b].double()
    return e - float(C)


def _pixels(d, nside):
    """RING pixels of directions d [n, 3] (FP64)."""
    N = nside
    r = d.norm(dim=1)
    z = d[:, 2] / r
    t = torch.remainder(torch.atan2(d[:, 1], d[:, 0]) * (2.0 / math.pi), 4.0)
    za = z.abs()
    jp = torch.floor(N * (0.5 + t - 0.75 * z)).long()
    jm = torch.floor(N * (0.5 + t + 0.75 * z)).long()
    ir = N + 1 + jp - jm
    ip = torch.div(jp + jm - N + 1 + (1 - (ir & 1)), 2, rounding_mode="floor") % (4 * N)
    belt = 2 * N * (N - 1) + (ir - 1) * 4 * N + ip
    s2 = (d[:, 0] ** 2 + d[:, 1] ** 2) / r ** 2
    tp = t - torch.floor(t)
    tmp = N * torch.sqrt(3.0 * s2 / (1.0 + za))
    ic = torch.floor(tp * tmp).long() + torch.floor((1.0 - tp) * tmp).long() + 1
    iq = torch.floor(t * ic).long() % (4 * ic)
    cap = torch.where(z > 0, 2 * ic * (ic - 1) + iq, 12 * N * N - 2 * ic * (ic + 1) + iq)
    return torch.where(za <= 2.0 / 3.0, belt, cap)


def _bin(xyz, boxes, chi, nside):
    npix = 12 * nside ** 2
    S = len(chi) - 1
    out = torch.zeros(S * npix, dtype=torch.int64, device=DEV)
    edges = torch.tensor(chi, dtype=torch.float64, device=DEV)
    for x, b in zip(xyz, boxes):
        d = x.double() - torch.tensor(list(b.obs), dtype=torch.float64, device=DEV)
        sh = torch.searchsorted(edges, d.norm(dim=1), right=True) - 1
        keep = (sh >= b.shell_lo) & (sh < b.shell_hi)
        out += torch.bincount(sh[keep] * npix + _pixels(d[keep], nside), minlength=S * npix)
    return out.view(S, npix)


def _statistics(counts, A, C, lo, hi):
    """(kappa, moments, statistics vector) of one realisation."""
    kap = _kappa(counts, A, C)
    k32 = kap.float().double()
    mom = _moments(k32)
    return kap, mom, torch.cat([mom[:6], _histogram(k32, lo, hi).double() / k32.numel()])


def _welford(v):
    mean = v.mean(dim=0)
    d = v - mean
    n = torch.full((1,), float(v.shape[0]), dtype=torch.float64, device=v.device)
    return torch.cat([n, mean, (d.T @ d).reshape(-1)])


def _rings(nside):
    """(first pixel, pixels, z, sin(theta), first azimuth) of every ring."""
    N, out = nside, []
    for i in range(1, 4 * N):
        k = min(i, 4 * N - i)
        if k < N:
            t = k * k / (3.0 * N * N)
            z, s = (1.0 - t), math.sqrt(t * (2.0 - t))
            start = 2 * k * (k - 1) if i < 2 * N else 12 * N * N - 2 * k * (k + 1)
            out.append((start, 4 * k, z if i < 2 * N else -z, s, math.pi / (4 * k)))
        else:
            z = 4.0 / 3.0 - 2.0 * i / (3.0 * N)
            out.append((2 * N * (N - 1) + 4 * N * (i - N), 4 * N, z, math.sqrt(1.0 - z * z),
                        ((i - N + 1) % 2) * math.pi / (4 * N)))
    return out


def _legendre(nside, lmax):
    """Yields (l, lambda_lm [l + 1, 2 nside] at the northern rings) for
    l = 0..lmax, the orthonormal Legendre functions by their recurrence in l.
    A value is kept as v 2^(800 e), e <= 0, so that sin^m does not vanish."""
    rings = _rings(nside)[:2 * nside]
    z = torch.tensor([r[2] for r in rings], dtype=torch.float64, device=DEV)
    sn = torch.tensor([r[3] for r in rings], dtype=torch.float64, device=DEV)
    P = 2 * nside
    big, small = 2.0 ** 400, 2.0 ** -800
    v1 = torch.zeros((lmax + 1, P), dtype=torch.float64, device=DEV)
    v2 = torch.zeros_like(v1)
    e = torch.zeros((lmax + 1, P), dtype=torch.int32, device=DEV)
    diag = torch.full((P,), math.sqrt(0.25 / math.pi), dtype=torch.float64, device=DEV)
    de = torch.zeros(P, dtype=torch.int32, device=DEV)
    m = torch.arange(lmax + 1, dtype=torch.float64, device=DEV)
    for l in range(lmax + 1):
        if l:
            diag = diag * sn * -math.sqrt((2 * l + 1) / (2.0 * l))
            low = diag.abs() < 1.0 / big
            diag = torch.where(low, diag / small, diag)
            de = de - low.int()
            mm = m[:l, None]
            a = torch.sqrt((4.0 * l * l - 1.0) / (l * l - mm * mm))
            b = torch.sqrt(((l - 1.0) ** 2 - mm * mm).clamp_(min=0.0) / (4.0 * (l - 1.0) ** 2 - 1.0))
            new = a * (z * v1[:l] - b * v2[:l])
            v2[:l] = v1[:l]
            v1[:l] = new
            if l % 16 == 0:
                up = (v1[:l].abs() > big) & (e[:l] < 0)
                v1[:l] = torch.where(up, v1[:l] * small, v1[:l])
                v2[:l] = torch.where(up, v2[:l] * small, v2[:l])
                e[:l] += up.int()
        v1[l], e[l] = diag, de
        yield l, torch.where(e[:l + 1] == 0, v1[:l + 1],
                             torch.where(e[:l + 1] == -1, v1[:l + 1] * small, 0.0))


def _map2alm(mp, nside, lmax):
    x = mp.double().cpu().numpy()
    rings = _rings(nside)
    m = np.arange(lmax + 1)
    F = np.empty((len(rings), lmax + 1), dtype=np.complex128)
    for i, (start, n, _, _, phi0) in enumerate(rings):
        F[i] = np.fft.fft(x[start:start + n])[m % n] * np.exp(-1j * phi0 * m)
    F = torch.from_numpy(F).to(DEV).T.contiguous()              # [m, ring]
    P = 2 * nside
    north, south = F[:, :P], F[:, P - 1:].flip(1).clone()       # ring r and its mirror
    south[:, P - 1] = 0.0                                       # the equator is its own
    even, odd = torch.view_as_real(north + south), torch.view_as_real(north - south)
    parts = [[even[..., 0].contiguous(), even[..., 1].contiguous()],
             [odd[..., 0].contiguous(), odd[..., 1].contiguous()]]
    out = torch.empty((lmax + 1) * (lmax + 2) // 2, dtype=torch.complex128, device=DEV)
    mi = torch.arange(lmax + 1, device=DEV)
    par = (mi & 1).bool()[:, None]
    both = [[torch.where(par, parts[1 - q][c], parts[q][c]) for c in range(2)] for q in range(2)]
    w = 4.0 * math.pi / (12.0 * nside * nside)
    for l, lam in _legendre(nside, lmax):
        f = both[l & 1]                                         # even or odd in l + m
        re, im = (lam * f[0][:l + 1]).sum(1), (lam * f[1][:l + 1]).sum(1)
        mm = mi[:l + 1]
        out[torch.div(mm * (2 * lmax + 1 - mm), 2, rounding_mode="floor") + l] = w * torch.complex(re, im)
    return out


def _alm2map(alm, nside, lmax):
    P = 2 * nside
    g = torch.zeros((2, 2, lmax + 1, P), dtype=torch.float64, device=DEV)   # [parity, re/im]
    mi = torch.arange(lmax + 1, device=DEV)
    for l, lam in _legendre(nside, lmax):
        mm = mi[:l + 1]
        a = alm[torch.div(mm * (2 * lmax + 1 - mm), 2, rounding_mode="floor") + l]
        for par in range(2):
            rows = slice(par, l + 1, 2)
            q = (l + par) & 1
            g[q, 0, rows] += a[rows].real[:, None] * lam[rows]
            g[q, 1, rows] += a[rows].imag[:, None] * lam[rows]
    north = torch.complex(g[0, 0] + g[1, 0], g[0, 1] + g[1, 1]).T.cpu().numpy()
    south = torch.complex(g[0, 0] - g[1, 0], g[0, 1] - g[1, 1]).T.cpu().numpy()
    out = np.empty(12 * nside * nside)
    m = np.arange(lmax + 1)
    for i, (start, n, _, _, phi0) in enumerate(_rings(nside)):
        G = (north[i] if i < P else south[4 * nside - 2 - i]) * np.exp(1j * phi0 * m)
        H = np.zeros(n, dtype=np.complex128)
        np.add.at(H, m % n, G)
        np.add.at(H, (-m[1:]) % n, G[1:].conj())
        out[start:start + n] = np.fft.ifft(H).real * n
    return torch.from_numpy(out).to(DEV)


def exact(case, seed):
    k = case["kind"]
    if k in ("bin", "periodic", "snapshots"):
        return None                                             # counts are whole numbers
    s = prepare(case, seed)
    if k == "kappa":
        kap = _kappa(s["counts"], s["A"], s["C"])
        return {"kappa": kap, "moments": _moments(kap.float().double()), "pdf": None}
    if k == "map":
        counts = _bin(s["xyz"], s["boxes"], s["chi"], s["nside"])
        kap, mom, vec = _statistics(counts, s["A"], s["C"], *s["range"])
        return {"counts": None, "kappa": kap, "moments": mom, "pdf": None, "vector": vec,
                "state": _welford(vec[None])}
    if k == "adjoint":
        e = _kappa(s["counts"], s["A"], s["C"])
        N = float(e.numel())
        d = e - e.mean()
        m2, m3 = (d ** 2).mean(), (d ** 3).mean()
        bar = 2.0 * d / N                                       # of the variance
        bar = bar + 3.0 / N * ((d * d - m2) / m2 ** 1.5 - m3 / m2 ** 2.5 * d)   # of the skewness
        if s["g"] is not None:
            bar = bar + s["g"].double()
        G = torch.stack([(bar * c.double()).sum() for c in s["counts"]]).cpu().numpy()
        grad = s["dA"] @ G - s["dC"] * float(bar.sum())
        if not s["fused"]:
            return {"grad": grad, "G": G}
        return {"kappa": e, "moments": _moments(e.float().double()), "pdf": None, "grad": grad,
                "G": G}
    if k == "spectrum":
        lmax = s["lmax"]
        alm = _map2alm(s["map"], s["nside"], lmax)
        l = _degrees(lmax)
        q = alm.abs() ** 2 * 2.0
        q[:lmax + 1] *= 0.5
        cl = torch.zeros(lmax + 1, dtype=torch.float64, device=DEV).index_add_(0, l, q)
        cl = cl / (2.0 * torch.arange(lmax + 1, device=DEV) + 1.0)
        nb = (lmax + 1 - 10) // 10
        return {"alm": alm, "cl": cl, "band": cl[10:10 + 10 * nb].view(nb, 10).mean(1)}
    if k == "smooth":
        l = _degrees(s["lmax"]).double()
        beam = torch.exp(-0.5 * l * (l + 1.0) * s["sigma"] ** 2)
        m = _alm2map(s["alm"] * beam, s["nside"], s["lmax"])
        return {"map": m, "moments": _moments(m.float().double()), "pdf": None}
    rows = [_statistics(_bin(x, b, s["chi"], s["nside"]), a, c, *s["range"])
            for x, b, a, c in zip(s["xyz"], s["boxes"], s["A"], s["C"])]
    vec = torch.stack([r[2] for r in rows])
    return {"moments": torch.stack([r[1] for r in rows]), "pdf": None, "vectors": vec,
            "state": _welford(vec)}
