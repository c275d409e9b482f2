"""Performance cases of the estimators: what programs measure, from the smallest call to the largest.

Every case goes through the public front end (``paper_2605_04864_gb300.api`` / ``.autograd``) on a
synthetic catalogue made on the GPU from the case's seed; ``exact`` evaluates the same definitions with
plain torch in float64.  Meshes, boxes, object numbers and bins are those of ``synthetic/configs.py``
and of the tests, with odd object and bin numbers among them.

Values of a mixed-precision measurement carry float32 accuracy and are kept as float32, as a program
stores its data vectors; FP64 measurements stay float64.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

DEV = "cuda"


# ---------------------------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------------------------
def _power(n, box, n_gal, n_ran, nbins, **kw):
    c = dict(kind="power", n=n, box=box, n_gal=n_gal, n_ran=n_ran, nbins=nbins, kmin=0.0, dk=0.01, ells="0,2,4",
             modified="", assign=3, interlace=1, precision="mixed", host=False)
    c.update(kw)
    return c


def _bispec(n, box, n_gal, n_ran, nbins, **kw):
    c = dict(kind="bispec", n=n, box=box, n_gal=n_gal, n_ran=n_ran, nbins=nbins, kmin=0.01, dk=0.01, scoc="0,2",
             tripo="0,2", shot="analytic", precision="mixed")
    c.update(kw)
    return c


def listed():
    return [
        # gradients inside an optimiser or a finite-difference check on a toy box: one small call, all latency
        dict(name="gradient_32", kind="gradient", n=32, box=93.75, n_gal=2_000, nbins=4, kmin=0.1, dk=0.1,
             precision="fp64"),
        # a small survey measured in double precision (validation runs): CIC, no interlacing
        dict(_power(64, 1000.0, 50_000, 500_000, 20, assign=2, interlace=0, precision="fp64"), name="power_fp64_64"),
        # one mock of a covariance set: a small survey, the standard multipoles
        dict(_power(128, 830.0, 123_457, 1_234_570, 48), name="power_128"),
        # a simulation box: periodic, global line of sight, odd number of objects
        dict(_power(256, 1000.0, 1_000_003, 0, 77), name="power_box_256"),
        # catalogues read from disk into host arrays and measured with the modified multipoles: the whole
        # call from host memory to host results
        dict(_power(256, 2000.0, 250_000, 2_500_000, 40, modified="4,6,8", host=True), name="power_host_256"),
        # the survey measurement at full size
        dict(_power(512, 2000.0, 2_000_000, 20_000_000, 80, modified="4,6,8"), name="power_512"),
        # two tracers of one survey: cross multipoles with the odd ones (relativistic dipole, octupole)
        dict(name="cross_192", kind="cross", n=192, box=1200.0, n_gal=211_111, n_gal_b=354_321, n_ran=2_111_110,
             n_ran_b=3_543_210, nbins=37, kmin=0.0, dk=0.01, ells="0,1,2,3,4", precision="mixed"),
        # bispectrum of a simulation box with the analytic shot noise
        dict(_bispec(256, 1000.0, 1_000_000, 0, 19), name="bispec_box_256"),
        # bispectrum of a survey: line of sight to each grid point, even and odd multipoles, raw
        dict(_bispec(128, 1000.0, 200_003, 2_000_030, 15, scoc="0,1,2,3", tripo="0", shot="raw"),
             name="bispec_survey_128"),
        # tri-polar bispectrum multipoles of a simulation box over every (k1, k2)
        dict(name="tripo_box_256", kind="tripo", n=256, box=1000.0, n_gal=1_000_000, nbins=19, kmin=0.01, dk=0.01,
             multipoles="000,110,112,202,220,222", precision="mixed"),
        # field-level inference: gradients of P_l and the equilateral B_0 with respect to the positions
        dict(name="gradient_1024", kind="gradient", n=1024, box=3000.0, n_gal=10_000_000, nbins=19, kmin=0.01, dk=0.01,
             precision="mixed"),
        # a handful of uneven mocks of a covariance set in one batch
        dict(name="batch_6", kind="batch", sizes="128,192,256,128,192,256", draw_seed=3000),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["gradient", "power_fp64", "power", "power", "power_box", "power_host", "cross", "bispec",
                       "bispec_survey", "tripo", "batch"])
    box = round(rng.uniform(500.0, 1500.0), 2)

    def pk_bins(n, b):
        return max(3, min(80, int(math.pi * n / b / 0.01 - 1e-9) - rng.randrange(3)))

    def bk_bins(n, b):   # from k = 0.01, below half the Nyquist wavenumber
        return max(3, min(19, int((0.5 * math.pi * n / b - 0.01) / 0.01 - 1e-9) - rng.randrange(3)))

    if kind == "gradient":
        n = rng.choice([32, 64, 96, 128, 192, 256, 512])
        b = n * 3000.0 / 1024
        # bins of 0.01 below k_N / 2 with the full mesh's resolution, wider ones on the small boxes
        dk = max(0.01, 1.5 * 2 * math.pi / b)
        nb = max(2, min(19, int((0.25 * 2 * math.pi / b * n - dk) / dk)))
        return dict(kind="gradient", n=n, box=b, n_gal=_logint(rng, 2_000, 40_000 * (n / 64) ** 2), nbins=nb, kmin=dk,
                    dk=dk, precision="fp64" if n <= 64 else "mixed")
    if kind == "power_fp64":
        n = rng.choice([32, 48, 64, 96, 128, 192])
        ng = _logint(rng, 5_000, 100_000)
        il = rng.randrange(2)
        return _power(n, box, ng, 10 * ng, pk_bins(n, box), assign=rng.choice([2, 3]), interlace=il, precision="fp64")
    if kind in ("power", "power_host"):
        n = rng.choice([64, 96, 128, 192, 256] if kind == "power_host" else [64, 96, 128, 192, 256, 512])
        box = round(box * max(1.0, n / 384), 2)
        ng = _logint(rng, 10_000 * (n / 64), 200_000 * (n / 128))
        return _power(n, box, ng, rng.choice([5, 10]) * ng, pk_bins(n, box), assign=rng.choice([2, 3, 3]),
                      ells=rng.choice(["0,2,4", "0,2"] + ["0,1,2,3,4"] * (n < 512)), modified=rng.choice(["", "4,6,8"]),
                      host=kind == "power_host")
    if kind == "power_box":
        n = rng.choice([64, 96, 128, 192, 256, 512])
        return _power(n, box, _logint(rng, 20_000, 2_000_000), 0, pk_bins(n, box), assign=rng.choice([2, 3, 3]),
                      interlace=rng.choice([0, 1, 1]))
    if kind == "cross":
        n = rng.choice([64, 96, 128, 192, 256])
        ga, gb = _logint(rng, 20_000, 400_000), _logint(rng, 20_000, 400_000)
        return dict(kind="cross", n=n, box=box, n_gal=ga, n_gal_b=gb, n_ran=10 * ga, n_ran_b=10 * gb,
                    nbins=pk_bins(n, box), kmin=0.0, dk=0.01, ells=rng.choice(["0,1,2,3,4", "0,2,4", "1,3"]),
                    precision="mixed")
    if kind == "bispec":
        n = rng.choice([64, 96, 128, 192, 256])
        b = round(rng.uniform(800.0, 1500.0), 2)
        return _bispec(n, b, _logint(rng, 50_000, 1_500_000), 0, bk_bins(n, b), shot=rng.choice(["analytic", "fft", "raw"]))
    if kind == "bispec_survey":
        n = rng.choice([64, 96, 128, 192])
        b = round(rng.uniform(800.0, 1500.0), 2)
        ng = _logint(rng, 20_000, 400_000)
        if rng.randrange(2):   # monopole with its shot noise, as the mocks of a batch take it
            return _bispec(n, b, ng, 10 * ng, bk_bins(n, b), scoc="0", tripo="0", shot=rng.choice(["analytic", "fft"]))
        return _bispec(n, b, ng, 10 * ng, bk_bins(n, b), scoc=rng.choice(["0,1,2,3", "0,2"]), tripo="0,2", shot="raw")
    if kind == "tripo":
        n = rng.choice([64, 96, 128, 192, 256])
        b = round(rng.uniform(800.0, 1500.0), 2)
        return dict(kind="tripo", n=n, box=b, n_gal=_logint(rng, 50_000, 1_500_000), nbins=bk_bins(n, b), kmin=0.01,
                    dk=0.01, multipoles=rng.choice(["000,202", "000,110,112,202,220,222", "220,222,224"]),
                    precision="mixed")
    sizes = [rng.choice([128, 192, 256]) for _ in range(rng.randint(2, 4))]
    return dict(kind="batch", sizes=",".join(str(s) for s in sizes), draw_seed=rng.randrange(1, 1 << 20))


def _ints(text):
    return tuple(int(v) for v in text.split(",")) if text else ()


def _multipoles(case):
    return [tuple(int(ch) for ch in mp) for mp in case["multipoles"].split(",")]


# ---------------------------------------------------------------------------------------------
# Inputs: clustered galaxies (lognormal) and uniform randoms, on the GPU, from the seed alone
# ---------------------------------------------------------------------------------------------
def _generator(seed, what=0):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1_000_003 + 7919 * what + 17) % (1 << 62))
    return g


def _lognormal(n_obj, box, n_gen, gen):
    """n_obj points of a lognormal field with P(k) ~ k^-1.5 (float64, cell by cell)."""
    kf = 2 * math.pi / box
    i = torch.fft.fftfreq(n_gen, 1.0 / n_gen, device=DEV)
    iz = torch.arange(n_gen // 2 + 1, device=DEV, dtype=torch.float32)
    k2 = i[:, None, None] ** 2 + i[None, :, None] ** 2 + iz[None, None, :] ** 2
    k2[0, 0, 0] = 1.0
    k = kf * k2.sqrt()
    mu2 = iz[None, None, :] ** 2 / k2
    amp = torch.sqrt(2.0e4 * (k / 0.05) ** -1.5 * torch.exp(-((k / 0.5) ** 2)) / (box / n_gen) ** 3) * (1 + 0.8 * mu2)
    amp[0, 0, 0] = 0.0
    white = torch.randn((n_gen,) * 3, device=DEV, generator=gen)
    dg = torch.fft.irfftn(torch.fft.rfftn(white) * amp, s=(n_gen,) * 3)
    lam = torch.exp(dg - 0.5 * dg.double().var().float()).reshape(-1)
    # integer intensities: their running sum does not depend on the order of additions
    c = torch.cumsum((lam / lam.max() * 2.0**30).to(torch.int64), 0)
    u = torch.randint(0, int(c[-1]), (n_obj,), device=DEV, generator=gen)
    cell = torch.searchsorted(c, u, right=True).sort().values
    pos = torch.stack([cell // (n_gen * n_gen), (cell // n_gen) % n_gen, cell % n_gen], 1).double()
    pos += torch.rand((n_obj, 3), device=DEV, generator=gen, dtype=torch.float64)
    return pos * (box / n_gen)


def _origin(box):
    """A cube whose centre lies 1.25 box sides from the observer along (1, 1, 1)."""
    return tuple(float(v) for v in (1.25 * box * np.ones(3) / math.sqrt(3.0) - 0.5 * box))


def _weights(n_obj, nbar, gen, dtype):
    """FKP weight times a completeness weight near 1."""
    w = 1.0 / (1.0 + nbar * 1.0e4) * (1.0 + 0.1 * (torch.rand(n_obj, device=DEV, generator=gen, dtype=torch.float64) - 0.5))
    return w.to(dtype)


def _catalog(n_obj, box, gen, dtype, n_gen=128, origin=None, clustered=True, nbar=None):
    if clustered:
        pos = _lognormal(n_obj, box, n_gen, gen)
    else:
        pos = torch.rand((n_obj, 3), device=DEV, generator=gen, dtype=torch.float64) * box
    nbar = n_obj / box**3 if nbar is None else nbar
    nb = torch.full((n_obj,), nbar, device=DEV, dtype=dtype)
    if origin is None:   # simulation box: unit weights
        return SimpleNamespace(pos=pos.to(dtype).contiguous(), w=torch.ones(n_obj, device=DEV, dtype=dtype), nbar=nb)
    pos += torch.tensor(origin, device=DEV, dtype=torch.float64)
    return SimpleNamespace(pos=pos.to(dtype).contiguous(), w=_weights(n_obj, nbar, gen, dtype), nbar=nb)


def _pair(case, seed, n_gal, n_ran, what=0):
    """(galaxies, randoms or None, origin) of one tracer."""
    dtype = torch.float64 if case.get("precision") == "fp64" else torch.float32
    gen = _generator(seed, what)
    n_gen = min(256, max(32, case["n"] // 2))
    box = case["box"]
    if n_ran == 0:
        return _catalog(n_gal, box, gen, dtype, n_gen), None, (0.0, 0.0, 0.0)
    o = _origin(box)
    g = _catalog(n_gal, box, gen, dtype, n_gen, o)
    return g, _catalog(n_ran, box, gen, dtype, origin=o, clustered=False, nbar=n_gal / box**3), o


def _batch_items(case, seed):
    """Uneven mocks: box sides U[500, 1500], galaxies log-uniform in [1e5, 2e6], ten times as many randoms, P_0,2,4 to the Nyquist wavenumber and B_0 below
    half of it."""
    shape = np.random.default_rng(case["draw_seed"])
    items = []
    for i, n in enumerate(_ints(case["sizes"])):
        box = float(shape.uniform(500.0, 1500.0))
        ng = int(round(math.exp(shape.uniform(math.log(1e5), math.log(2e6)))))
        kn = math.pi * n / box
        g, r, o = _pair(dict(n=n, box=box), seed, ng, 10 * ng, what=i)
        items.append(dict(n=n, box=box, data=g, randoms=r, origin=o,
                          power_bins=(0.0, 0.01, min(80, int(math.floor(kn / 0.01 - 1e-9)))),
                          bispec_bins=(0.01, 0.01, min(19, int(math.floor((0.5 * kn - 0.01) / 0.01 - 1e-9))))))
    return items


def _kbins(case):
    return (case["kmin"], case["dk"], case["nbins"])


def _cotangents(case, seed):
    """Cotangents of P_0,2,4 and B_0 as a likelihood's backward pass hands them over."""
    gen = _generator(seed, 99)
    nb = case["nbins"]
    gp = torch.randn((3, nb), device=DEV, generator=gen, dtype=torch.float64) * 1e-4
    gb = torch.randn((nb,), device=DEV, generator=gen, dtype=torch.float64) * 1e-9
    return gp, gb


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    f64 = dict(device=DEV, dtype=torch.float64)
    if kind == "power":
        g, r, st["origin"] = _pair(case, seed, case["n_gal"], case["n_ran"])
        if case["host"]:
            g, r = (SimpleNamespace(**{k: v.cpu().numpy() for k, v in vars(c).items()}) for c in (g, r))
        else:
            rows = 2 + len(_ints(case["ells"])) + len(_ints(case["modified"]))
            st["out"] = torch.zeros(rows * case["nbins"] + 8, **f64)
        st["data"], st["randoms"] = g, r
    elif kind == "cross":
        st["a"], st["ra"], st["origin"] = _pair(case, seed, case["n_gal"], case["n_ran"])
        st["b"], st["rb"], _ = _pair(case, seed, case["n_gal_b"], case["n_ran_b"], what=1)
        st["out"] = torch.zeros((2 + len(_ints(case["ells"]))) * case["nbins"] + 8, **f64)
    elif kind == "bispec":
        st["data"], st["randoms"], st["origin"] = _pair(case, seed, case["n_gal"], case["n_ran"])
        st["out"] = torch.zeros(sum(size for _, size in _bispec_layout(case)), **f64)
    elif kind == "tripo":
        st["data"], _, _ = _pair(case, seed, case["n_gal"], 0)
        nb = case["nbins"]
        st["out"] = torch.zeros(2 * len(_multipoles(case)) * nb * nb + nb + 8, **f64)
    elif kind == "gradient":
        g, _, _ = _pair(case, seed, case["n_gal"], 0)
        st["pos"] = g.pos.requires_grad_(True)
        st["gp"], st["gb"] = _cotangents(case, seed)
    else:
        from paper_2605_04864_gb300 import api

        st["items"] = _batch_items(case, seed)
        st["arr"], st["keep"] = api.make_batch(st["items"])
        total, _ = api.batch_layout(st["arr"])
        st["out"] = torch.zeros(total, **f64)
    return st


# ---------------------------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------------------------
_SHOT = {"raw": False, "analytic": True, "fft": "fft"}


def _triangles(nb, kmin, dk):
    c = [kmin + (b + 0.5) * dk for b in range(nb)]
    return [(i, j, k) for i in range(nb) for j in range(i, nb) for k in range(j, nb) if c[k] <= c[i] + c[j] + 1e-9 * dk]


def _pairs(nb):
    return [(i, j) for i in range(nb) for j in range(i, nb)]


def _bispec_layout(case):
    nt, npair = len(_triangles(case["nbins"], case["kmin"], case["dk"])), len(_pairs(case["nbins"]))
    sc, tr = _ints(case["scoc"]), _ints(case["tripo"])
    return ([(f"B{l}", nt) for l in sc] + [(f"shot_B{l}", nt) for l in sc] + [("NT", nt)]
            + [(f"B{l}0{l}", npair) for l in tr] + [(f"shot_B{l}0{l}", npair) for l in tr]
            + [("nmodes", case["nbins"]), ("scalars", 8)])


def _power_layout(case):
    nb = case["nbins"]
    return ([("k", nb), ("nmodes", nb)] + [(f"P{l}", nb) for l in _ints(case["ells"])]
            + [(f"P{l}b", nb) for l in _ints(case.get("modified", ""))] + [("scalars", 8)])


def _tripo_layout(case):
    nb = case["nbins"]
    names = ["".join(str(v) for v in mp) for mp in _multipoles(case)]
    return [(f"B{v}", nb * nb) for v in names] + [(f"shot_B{v}", nb * nb) for v in names] + [("nmodes", nb), ("scalars", 8)]


def _named(flat, layout):
    out, o = {}, 0
    for name, size in layout:
        out[name] = flat[o:o + size]
        o += size
    return out


def run(state):
    from paper_2605_04864_gb300 import api, autograd

    c = state["case"]
    kind = c["kind"]
    if kind == "gradient":
        n, vol = c["n_gal"], c["box"] ** 3
        pos = state["pos"]
        mesh = autograd.paint(pos, None, c["n"], c["box"], precision=c["precision"])
        r = autograd.mesh_multipoles(mesh, c["box"], _kbins(c), i22=n * n / vol, n0=vol / n, i33=n**3 / vol**2,
                                     precision=c["precision"])
        (grad,) = torch.autograd.grad([r["P"], r["B0"]], [pos], [state["gp"], state["gb"]])
        keep = grad.dtype
        return {"P": r["P"].detach().to(keep), "B0": r["B0"].detach().to(keep), "NT": r["NT"].to(keep), "grad": grad}
    if kind == "batch":
        return {"out": api.batch_run(state["arr"], state["out"]).float()}
    common = dict(n=c["n"], box=c["box"], kbins=_kbins(c), precision=c["precision"])
    if kind == "power":
        layout = _power_layout(c)
        common.update(assign=c["assign"], interlace=c["interlace"], ells=_ints(c["ells"]),
                      modified=_ints(c["modified"]), origin=state["origin"],
                      los_dir=(0.0, 0.0, 1.0) if state["randoms"] is None else None)
        if c["host"]:
            r = api.power_multipoles(state["data"], state["randoms"], **common)
            flat = np.concatenate([r["k_eff"], r["nmodes"], *r["P"].values(), *r["Pmod"].values(),
                                   np.array(list(r["scalars"].values()))])
            return _named(flat.astype(np.float32), layout)
        flat = api.power_multipoles(state["data"], state["randoms"], out=state["out"], **common)
    elif kind == "cross":
        layout = _power_layout(c)
        flat = api.cross_power_multipoles(state["a"], state["ra"], state["b"], state["rb"], ells=_ints(c["ells"]),
                                          origin=state["origin"], out=state["out"], **common)
    elif kind == "bispec":
        layout = _bispec_layout(c)
        flat = api.bispectrum(state["data"], randoms=state["randoms"], scoc_ells=_ints(c["scoc"]),
                              tripo_ells=_ints(c["tripo"]), shot=_SHOT[c["shot"]], origin=state["origin"],
                              los_dir=(0.0, 0.0, 1.0) if state["randoms"] is None else None, out=state["out"], **common)
    else:
        layout = _tripo_layout(c)
        flat = api.bispectrum_sugiyama(state["data"], multipoles=_multipoles(c), out=state["out"], **common)
    return _named(flat if c["precision"] == "fp64" else flat.float(), layout)


# ---------------------------------------------------------------------------------------------
# What a pass cannot do without: the catalogues read once, the results written once, the transforms of
# the fields the estimator is made of (2.5 n^3 log2 n^3 each, real) and the triple-product sums.
# ---------------------------------------------------------------------------------------------
def _fft_flops(n, fields):
    return fields * 2.5 * n**3 * 3 * math.log2(n)


def _fields(ells):
    return sum(2 * l + 1 for l in set(ells) | {0})


def _shell_grid(case):
    """Points per side that hold the closed triples of the largest bin without aliasing."""
    return math.floor(3 * (case["kmin"] + case["nbins"] * case["dk"]) * case["box"] / (2 * math.pi)) + 1


def work(case):
    kind = case["kind"]
    if kind == "batch":
        tot = {"bytes": 0.0, "flops": 0.0}
        shape = np.random.default_rng(case["draw_seed"])
        for n in _ints(case["sizes"]):
            box = float(shape.uniform(500.0, 1500.0))
            ng = int(round(math.exp(shape.uniform(math.log(1e5), math.log(2e6)))))
            kn = math.pi * n / box
            nb = min(19, int(math.floor((0.5 * kn - 0.01) / 0.01 - 1e-9)))
            for w in (work(_power(n, box, ng, 10 * ng, min(80, int(kn / 0.01)))),
                      work(_bispec(n, box, 0, 0, nb, scoc="0", tripo=""))):
                tot["bytes"] += w["bytes"]
                tot["flops"] += w["flops"]
        return tot
    es = 8 if case["precision"] == "fp64" else 4
    n, nb = case["n"], case["nbins"]
    objects = case["n_gal"] + case.get("n_ran", 0) + case.get("n_gal_b", 0) + case.get("n_ran_b", 0)
    if kind == "gradient":
        # positions read, gradients written; the mesh's transforms and, per bin, the shell field, its
        # square's transform and the gradient's share on the grid the triples need
        return {"bytes": 6.0 * es * objects + 8.0 * 5 * nb,
                "flops": _fft_flops(n, 2) + _fft_flops(min(n, _shell_grid(case)), 3 * nb)}
    bytes_ = 5.0 * es * objects
    if kind in ("power", "cross"):
        ells = set(_ints(case["ells"])) | ({2, 4} if case.get("modified") else set())
        fields = 1 if not case.get("n_ran", 0) else _fields(ells)
        phases = 2 if case.get("interlace", 1) else 1
        return {"bytes": bytes_ + 8.0 * (nb * (2 + len(ells) + len(_ints(case.get("modified", "")))) + 8),
                "flops": _fft_flops(n, phases * (fields + (1 if kind == "cross" else 0)))}
    ns = min(n, _shell_grid(case))
    if kind == "tripo":
        mps = _multipoles(case)
        shells = {(l, m) for l1, l2, _ in mps for l in (l1, l2) for m in range(min(l1, l2) + 1)}
        parts = sum(1 if m == 0 else 2 for _, m in shells)
        prods = sum((1 if m == 0 else 2) for l1, l2 in {(a, b) for a, b, _ in mps} for m in range(min(l1, l2) + 1))
        return {"bytes": bytes_ + 8.0 * (2 * len(mps) * nb * nb + nb + 8),
                "flops": _fft_flops(n, 2) + _fft_flops(ns, parts * nb + 1) + 2.0 * prods * nb * nb * ns**3}
    scoc, tripo = _ints(case["scoc"]), _ints(case["tripo"])
    fields = 2 * _fields(scoc + tripo) if case["n_ran"] and set(scoc + tripo) != {0} else 2
    if case["shot"] != "raw":
        fields += 2
    families = len(set(scoc) | {0})
    sums = len(scoc) * len(_triangles(nb, case["kmin"], case["dk"])) + len(tripo) * len(_pairs(nb))
    return {"bytes": bytes_ + 8.0 * sum(s for _, s in _bispec_layout(case)),
            "flops": _fft_flops(n, fields) + _fft_flops(ns, families * nb + len(tripo)) + 3.0 * sums * ns**3}


# ---------------------------------------------------------------------------------------------
# The same values in float64 with plain torch
# ---------------------------------------------------------------------------------------------
def _scalars(d, r, box):
    w = d.w.double()
    if r is None:
        ws, vol = w.sum(), box**3
        i22 = ws * ws / vol
        return dict(alpha=0.0 * ws, I22=i22, I33=ws**3 / vol**2, N0=(w * w).sum() / i22, S3=(w**3).sum(), wg=ws,
                    wr=0.0 * ws, w2=(w * w).sum())
    wr, nb = r.w.double(), r.nbar.double()
    a = w.sum() / wr.sum()
    i22 = a * (nb * wr * wr).sum()
    w2 = (w * w).sum() + a * a * (wr * wr).sum()
    return dict(alpha=a, I22=i22, I33=a * (nb * nb * wr**3).sum(), N0=w2 / i22,
                S3=(w**3).sum() - a**3 * (wr**3).sum(), wg=w.sum(), wr=wr.sum(), w2=w2)


def _scalar_vec(sc):
    return torch.stack([sc[k] for k in ("alpha", "I22", "I33", "N0", "S3", "wg", "wr", "w2")])


def _taps(s, assign):
    """Base cell and per-tap weights (and their derivatives) along each axis."""
    if assign == 2:
        i0 = torch.floor(s)
        d = s - i0
        return i0.long(), ((0, 1.0 - d, None), (1, d, None))
    i0 = torch.floor(s + 0.5)
    d = s - i0
    return i0.long(), ((-1, 0.5 * (0.5 - d) ** 2, d - 0.5), (0, 0.75 - d * d, -2.0 * d), (1, 0.5 * (0.5 + d) ** 2, d + 0.5))


def _paint(mesh, pos, w, n, box, origin, assign, shift):
    o = torch.tensor(origin, device=DEV, dtype=torch.float64)
    flat = mesh.view(-1)
    for p, ww in zip(pos.split(1 << 22), w.split(1 << 22)):
        i0, taps = _taps((p.double() - o) * (n / box) + shift, assign)
        for ox, wx, _ in taps:
            for oy, wy, _ in taps:
                ixy = ((i0[:, 0] + ox) % n * n + (i0[:, 1] + oy) % n) * n
                wxy = ww * wx[:, 0] * wy[:, 1]
                for oz, wz, _ in taps:
                    flat.index_add_(0, ixy + (i0[:, 2] + oz) % n, wxy * wz[:, 2])


def _meshes(d, r, sc, n, box, origin, assign, interlace, power=1):
    out = []
    for ph in range(2 if interlace else 1):
        m = torch.zeros((n,) * 3, device=DEV, dtype=torch.float64)
        _paint(m, d.pos, d.w.double() ** power, n, box, origin, assign, 0.5 * ph)
        if r is not None:
            coef = -sc["alpha"] if power == 1 else sc["alpha"] ** 2
            _paint(m, r.pos, coef * r.w.double() ** power, n, box, origin, assign, 0.5 * ph)
        elif power == 1:
            m -= sc["wg"] / float(n) ** 3
        out.append(m)
    return out


def _axis(n):
    return torch.fft.fftfreq(n, 1.0 / n, device=DEV, dtype=torch.float64)


def _modes(n):
    """Integer wavevectors of the half grid (x, y, z >= 0)."""
    i = _axis(n)
    return i[:, None, None], i[None, :, None], torch.arange(n // 2 + 1, device=DEV, dtype=torch.float64)[None, None, :]


def _bins(n, box, kbins):
    """Bin of each half-grid mode (-1: none), its |k| and its weight (modes k and -k)."""
    i, j, l = _modes(n)
    k = (2 * math.pi / box) * (i * i + j * j + l * l).sqrt()
    b = torch.floor((k - kbins[0]) / kbins[1])
    ok = (b >= 0) & (b < kbins[2]) & (k > 0) & (i != -n // 2) & (j != -n // 2) & (l != n // 2)
    return torch.where(ok, b, -1.0).long(), k, torch.where(l > 0, 2.0, 1.0).expand_as(k)


def _binsum(v, b, nb):
    return torch.bincount((b + 1).reshape(-1), weights=v.reshape(-1), minlength=nb + 1)[1:nb + 1]


def _spectrum(parts, n, assign):
    """Interlaced, compensated spectrum from the one or two phases' transforms."""
    i, j, l = _modes(n)
    s = parts[0]
    if len(parts) == 2:
        s = 0.5 * (s + torch.exp(1j * math.pi * (i + j + l) / n) * parts[1])
    for a in (i, j, l):
        s = s / torch.sinc(a / n) ** assign
    return s


def _harmonics(l, x, y, z):
    """2l+1 real functions R of a unit vector with sum R(u) R(v) = L_l(u.v)."""
    leg = np.polynomial.legendre.leg2poly([0.0] * l + [1.0])
    for m in range(l + 1):
        poly = np.polynomial.polynomial.polyder(leg, m) if m else leg
        c = math.sqrt((1 if m == 0 else 2) * math.factorial(l - m) / math.factorial(l + m))
        q = torch.zeros_like(z)
        for a in poly[::-1]:
            q = q * z + float(a)
        re, im = torch.ones_like(x + y), torch.zeros_like(x + y)
        for _ in range(m):
            re, im = re * x - im * y, re * y + im * x
        yield c * q * re
        if m:
            yield c * q * im


def _unit(x, y, z):
    inv = 1.0 / (x * x + y * y + z * z).sqrt().clamp_min(1e-300)
    return x * inv, y * inv, z * inv


def _yamamoto(meshes, ells, n, box, origin, assign):
    """{l: F_l(k)}: line of sight from the observer (at 0) to each grid point."""
    out = {0: _spectrum([torch.fft.rfftn(m) for m in meshes], n, assign)}
    ku = _unit(*_modes(n))
    ku[2][0, 0, 0] = 1.0   # the zero mode's direction is taken along z
    g = torch.arange(n, device=DEV, dtype=torch.float64)
    for l in ells:
        if l == 0:
            continue
        xs = []
        for ph in range(len(meshes)):
            a = [o + (g - 0.5 * ph) * (box / n) for o in origin]
            xs.append(_unit(a[0][:, None, None], a[1][None, :, None], a[2][None, None, :]))
        gens = [_harmonics(l, *u) for u in xs]
        acc = 0.0
        for kk in _harmonics(l, *ku):
            acc = acc + kk * _spectrum([torch.fft.rfftn(m * next(gx)) for m, gx in zip(meshes, gens)], n, assign)
        out[l] = acc
    return out


def _legendre(l, mu):
    return (torch.ones_like(mu), mu, 1.5 * mu * mu - 0.5, 2.5 * mu**3 - 1.5 * mu, (35 * mu**4 - 30 * mu * mu + 3) / 8)[l]


def _mu_z(n):
    i, j, l = _modes(n)
    k = (i * i + j * j + l * l).sqrt()
    return l / k.clamp_min(1e-300)


def _exact_power(d, r, case, origin, ells, modified):
    n, box, kb, nb = case["n"], case["box"], _kbins(case), case["nbins"]
    sc = _scalars(d, r, box)
    meshes = _meshes(d, r, sc, n, box, origin, case["assign"], case["interlace"])
    need = sorted(set(ells) | {0} | ({2, 4} if modified else set()))
    if r is None:
        f0 = _spectrum([torch.fft.rfftn(m) for m in meshes], n, case["assign"])
        f = {l: _legendre(l, _mu_z(n)) * f0 for l in need}
    else:
        f = _yamamoto(meshes, need, n, box, origin, case["assign"])
    b, k, wt = _bins(n, box, kb)
    cnt = _binsum(wt, b, nb)
    div = cnt.clamp_min(1.0)

    def mean(x, y, odd=False):
        v = x * y.conj()
        return _binsum(wt * (v.imag if odd else v.real), b, nb) / div

    p = {l: torch.where(cnt > 0, (2 * l + 1) / sc["I22"] * mean(f[0], f[l], l % 2 == 1) - (sc["N0"] if l == 0 else 0.0), 0.0)
         for l in need}
    out = {"k": torch.where(cnt > 0, _binsum(wt * k, b, nb) / div, 0.0), "nmodes": cnt}
    out.update({f"P{l}": p[l] for l in ells})
    if modified:
        p22 = 9 / sc["I22"] * mean(f[2], f[2]) - 9.0 / 5 * sc["N0"]
        p42 = 13 / sc["I22"] * mean(f[4], f[2])
        p44 = 17 / sc["I22"] * mean(f[4], f[4]) - 17.0 / 9 * sc["N0"]
        pm = {4: 35 / 18 * p22 - p[2] - 3.5 * p[0], 6: 11 / 5 * p42 - 52 / 63 * p[4] - 286 / 175 * p[2],
              8: 1287 / 490 * p44 - 374 / 245 * p42 - 3553 / 15435 * p[4] - 1326 / 8575 * p[2] - 2431 / 490 * p[0]}
        out.update({f"P{l}b": torch.where(cnt > 0, pm[l], 0.0) for l in modified})
    out["scalars"] = _scalar_vec(sc)
    return out


def _exact_cross(case, seed):
    n, box, kb, nb, ells = case["n"], case["box"], _kbins(case), case["nbins"], _ints(case["ells"])
    a, ra, o = _pair(case, seed, case["n_gal"], case["n_ran"])
    bb, rb, _ = _pair(case, seed, case["n_gal_b"], case["n_ran_b"], what=1)
    sa, sb = _scalars(a, ra, box), _scalars(bb, rb, box)
    fa = _yamamoto(_meshes(a, ra, sa, n, box, o, 3, 1), (0,), n, box, o, 3)[0]
    fb = _yamamoto(_meshes(bb, rb, sb, n, box, o, 3, 1), ells, n, box, o, 3)
    b, k, wt = _bins(n, box, kb)
    cnt = _binsum(wt, b, nb)
    div = cnt.clamp_min(1.0)
    i22 = (sa["I22"] * sb["I22"]).sqrt()
    out = {"k": torch.where(cnt > 0, _binsum(wt * k, b, nb) / div, 0.0), "nmodes": cnt}
    for l in ells:
        v = fa * fb[l].conj()
        out[f"P{l}"] = (2 * l + 1) / i22 * _binsum(wt * (v.imag if l % 2 else v.real), b, nb) / div
    out["scalars"] = torch.stack([sa["alpha"], i22, sb["alpha"], 0.0 * i22, sa["I22"], sb["I22"], sa["wg"], sb["wg"]])
    return out


def _real(x, n):
    """sum_q x(q) e^{iq.x} on the n grid."""
    return torch.fft.irfftn(x, s=(n,) * 3) * float(n) ** 3


def _shells(x, b, nb, n):
    return torch.stack([_real(torch.where(b == i, x, 0.0), n).reshape(-1) for i in range(nb)])


def _triple(fi, fj, fk, tri, n):
    """sum_x fi_i fj_j fk_k / n^3 over the triangles (grouped by (i, j))."""
    out, by = torch.zeros(len(tri), device=DEV, dtype=torch.float64), {}
    for t, (i, j, k) in enumerate(tri):
        by.setdefault((i, j), []).append((t, k))
    for (i, j), tk in by.items():
        k0, k1 = tk[0][1], tk[-1][1] + 1
        s = fk[k0:k1] @ (fi[i] * fj[j])
        out[torch.tensor([t for t, _ in tk], device=DEV)] = s[torch.tensor([k - k0 for _, k in tk], device=DEV)]
    return out / float(n) ** 3


def _pair_sums(fi, fj, g, n):
    p = torch.stack([fi[i] * g for i in range(len(fi))]) @ fj.T / float(n) ** 3
    return torch.stack([p[i, j] for i, j in _pairs(len(fi))])


def _g_ring(l, t):
    """The ring factor of the compressed shot noise, by quadrature of its integral form."""
    x, w = np.polynomial.legendre.leggauss(400)
    lo, hi = abs(t - 1.0), t + 1.0
    x = 0.5 * (hi - lo) * x + 0.5 * (hi + lo)
    leg = np.polynomial.legendre.legval((x * x + t * t - 1.0) / (2.0 * x * t), [0.0] * l + [1.0])
    return float(0.5 * (hi - lo) * np.sum(w * x * leg) / (2.0 * t))


def _exact_bispec(d, r, case, origin, assign=3):
    n, box, kb, nb = case["n"], case["box"], _kbins(case), case["nbins"]
    scoc, tripo = _ints(case["scoc"]), _ints(case["tripo"])
    kmin, dk, _ = kb
    cen = [kmin + (q + 0.5) * dk for q in range(nb)]
    tri, prs = _triangles(nb, kmin, dk), _pairs(nb)
    sc = _scalars(d, r, box)
    i33, s3 = sc["I33"], sc["S3"]
    ells = sorted(set(scoc) | set(tripo) | {0})
    x = _yamamoto(_meshes(d, r, sc, n, box, origin, assign, 1), ells if r is not None else (0,), n, box, origin, assign)
    if r is None:
        x = {l: _legendre(l, _mu_z(n)) * x[0] for l in ells}
    b, kmag, wt = _bins(n, box, kb)
    cnt = _binsum(wt, b, nb)
    one = torch.ones_like(x[0])
    i, j, l_ = _modes(n)
    inside = (kmag < 2.0001 * (kmin + nb * dk)) & (i != -n // 2) & (j != -n // 2) & (l_ != n // 2)
    f0, ind = _shells(x[0], b, nb, n), _shells(one, b, nb, n)
    nt = torch.round(_triple(ind, ind, ind, tri, n))
    ntd = nt.clamp_min(1.0)
    raw, comp, shot, cshot = {}, {}, {}, {}
    for l in scoc:
        fl = f0 if l == 0 else _shells(x[l] if l % 2 == 0 else -1j * x[l], b, nb, n)
        raw[l] = torch.where(nt > 0, (2 * l + 1) / i33 * _triple(fl, f0, f0, tri, n) / ntd, 0.0)
        shot[l] = torch.zeros_like(raw[l])
        del fl
    nij = torch.stack([cnt[i_] * cnt[j_] for i_, j_ in prs])
    for l in tripo:
        g = _real(torch.where(inside, x[l], 0.0), n).reshape(-1)
        comp[l] = torch.where(nij > 0, (2 * l + 1) / i33 * _pair_sums(f0, f0, g, n) / nij.clamp_min(1.0), 0.0)
        cshot[l] = torch.zeros_like(comp[l])
    if case["shot"] != "raw":
        xn_mesh = _meshes(d, r, sc, n, box, origin, assign, 1, power=2)
        xn = x[0] * _yamamoto(xn_mesh, (0,), n, box, origin, assign)[0].conj()
    if case["shot"] == "analytic":
        del f0, ind
        nq = int(math.ceil(2.0 * (kmin + nb * dk) / dk)) + 1
        bq, _, _ = _bins(n, box, (0.0, dk, nq))

        def term(l, bb, m):
            lmu = _legendre(l, _mu_z(n)).expand_as(wt)
            c = _binsum(wt, bb, m)
            v = (_binsum(wt * lmu * xn.real, bb, m) - s3 * _binsum(wt * lmu, bb, m)) / c.clamp_min(1.0)
            return v.tolist(), c.tolist()

        for l in sorted(set(scoc) | set(tripo)):
            h, _ = term(l, b, nb)
            q, cq = term(l, bq, nq)
            s0 = float(s3) if l == 0 else 0.0
            pl = lambda v: float(np.polynomial.legendre.legval(v, [0.0] * l + [1.0]))  # noqa: E731
            if l in scoc:
                v = []
                for a, e, f in tri:
                    c12 = (cen[f] ** 2 - cen[a] ** 2 - cen[e] ** 2) / (2 * cen[a] * cen[e])
                    c13 = (cen[e] ** 2 - cen[a] ** 2 - cen[f] ** 2) / (2 * cen[a] * cen[f])
                    v.append(s0 + h[a] + pl(c12) * h[e] + pl(c13) * h[f])
                shot[l] = (2 * l + 1) / i33 * torch.tensor(v, device=DEV, dtype=torch.float64)
            if l in tripo:
                v = []
                for a, e in prs:
                    t = s0 + _g_ring(l, cen[a] / cen[e]) * h[a] + _g_ring(l, cen[e] / cen[a]) * h[e]
                    lo, hi = abs(cen[a] - cen[e]) + 0.5 * dk, cen[a] + cen[e] - 0.5 * dk
                    m = [(cq[s] / ((s + 0.5) * dk), q[s]) for s in range(nq)
                         if lo - 1e-9 * dk <= (s + 0.5) * dk <= hi + 1e-9 * dk and cq[s] > 0]
                    v.append(t + (sum(w * y for w, y in m) / sum(w for w, _ in m) if m else 0.0))
                cshot[l] = (2 * l + 1) / i33 * torch.tensor(v, device=DEV, dtype=torch.float64)
    elif case["shot"] == "fft":
        dn = _shells(xn, b, nb, n)
        for l in scoc:
            lmu = _legendre(l, _mu_z(n)) if l else one.real
            dl, il = (dn, ind) if l == 0 else (_shells(lmu * xn, b, nb, n), _shells(lmu * one, b, nb, n))
            t = (_triple(dl, ind, ind, tri, n) + _triple(il, dn, ind, tri, n) + _triple(il, ind, dn, tri, n)
                 - 2 * s3 * _triple(il, ind, ind, tri, n))
            shot[l] = torch.where(nt > 0, (2 * l + 1) / i33 * t / ntd, 0.0)
        for l in tripo:
            lmu = _legendre(l, _mu_z(n)) if l else one.real
            gd = _real(torch.where(inside, lmu * xn, 0.0), n).reshape(-1)
            gl = _real(torch.where(inside, lmu * one, 0.0), n).reshape(-1)
            t = (_pair_sums(ind, ind, gd - 2 * s3 * gl, n) + _pair_sums(ind, dn, gl, n) + _pair_sums(dn, ind, gl, n))
            cshot[l] = torch.where(nij > 0, (2 * l + 1) / i33 * t / nij.clamp_min(1.0), 0.0)
    out = {f"B{l}": torch.where(nt > 0, raw[l] - shot[l], 0.0) for l in scoc}
    out.update({f"shot_B{l}": shot[l] for l in scoc})
    out["NT"] = nt
    out.update({f"B{l}0{l}": comp[l] - cshot[l] for l in tripo})
    out.update({f"shot_B{l}0{l}": cshot[l] for l in tripo})
    out["nmodes"], out["scalars"] = cnt, _scalar_vec(sc)
    return out


def _wigner3j(a, b, c, m1, m2, m3):
    f = math.factorial
    if m1 + m2 + m3 or abs(m1) > a or abs(m2) > b or abs(m3) > c or not abs(a - b) <= c <= a + b:
        return 0.0
    tri = f(a + b - c) * f(a - b + c) * f(-a + b + c) / f(a + b + c + 1)
    s = 0.0
    for k in range(a + b + c + 1):
        den = (k, a + b - c - k, a - m1 - k, b + m2 - k, c - b + m1 + k, c - a - m2 + k)
        if min(den) >= 0:
            s += (-1) ** k / math.prod(f(v) for v in den)
    norm = math.prod(f(v) for v in (a + m1, a - m1, b + m2, b - m2, c + m3, c - m3))
    return (-1) ** (a - b - m3) * math.sqrt(tri * norm) * s


def _exact_tripo(case, seed):
    n, box, nb = case["n"], case["box"], case["nbins"]
    d, _, o = _pair(case, seed, case["n_gal"], 0)
    sc = _scalars(d, None, box)
    x = _yamamoto(_meshes(d, None, sc, n, box, o, 3, 1), (0,), n, box, o, 3)[0]
    b, kmag, wt = _bins(n, box, _kbins(case))
    cnt = _binsum(wt, b, nb)
    i, j, l_ = _modes(n)
    inside = (kmag < 2.0001 * (case["kmin"] + nb * case["dk"])) & (i != -n // 2) & (j != -n // 2) & (l_ != n // 2)
    g = _real(torch.where(inside, x, 0.0), n).reshape(-1)
    kx, ky, kz = _unit(*_modes(n))
    cache = {}

    def shells(l, m):
        """Real and imaginary parts of F_l^m = sum_q e^{iqx} y_l^{m*} X (Condon-Shortley phase, Racah norm)."""
        if (l, m) not in cache:
            h = list(_harmonics(l, kx, ky, kz))
            c = (-1) ** m / math.sqrt(2.0) if m else 1.0
            re = c * h[max(0, 2 * m - 1)]
            im = c * h[2 * m] if m else torch.zeros_like(re)
            # y real and imaginary parts have the parity of l: even weights give real fields, odd ones i times real
            even = l % 2 == 0
            fr = _shells(re * x if even else -1j * re * x, b, nb, n)
            fi = _shells(im * x if even else -1j * im * x, b, nb, n) if m else torch.zeros_like(fr)
            # even: F = fr - i fi; odd: F = i fr + fi
            cache[(l, m)] = (fr, -fi) if even else (fi, fr)
        return cache[(l, m)]

    out = {}
    div = (cnt[:, None] * cnt[None, :]).clamp_min(1.0)
    for l1, l2, ll in _multipoles(case):
        acc = torch.zeros((nb, nb), device=DEV, dtype=torch.float64)
        for m in range(min(l1, l2) + 1):
            ar, ai = shells(l1, m)
            br, bi = shells(l2, m)
            # F_l2^{-m} = (-1)^{l2+m} conj(F_l2^m); m and -m together give twice the real part
            w = _wigner3j(l1, l2, ll, m, -m, 0) * (-1) ** (l2 + m) * (2 if m else 1)
            acc += w * ((ar * g) @ br.T + (ai * g) @ bi.T) / float(n) ** 3
        hn = _wigner3j(l1, l2, ll, 0, 0, 0) * (2 * l1 + 1) * (2 * l2 + 1) * (2 * ll + 1)
        v = torch.where(cnt[:, None] * cnt[None, :] > 0, hn * acc / (sc["I33"] * div), 0.0)
        out[f"B{l1}{l2}{ll}"] = v.reshape(-1)
    out.update({f"shot_{k}": torch.zeros_like(v) for k, v in list(out.items())})
    out["nmodes"], out["scalars"] = cnt, _scalar_vec(sc)
    return out


def _coarse(x, n, m):
    """The half-grid spectrum x (n grid) cut to the m grid's modes (m <= n, its Nyquist planes zero)."""
    h = m // 2
    idx = torch.tensor(list(range(h)) + [0] + list(range(n - h + 1, n)), device=DEV)
    y = x[idx][:, idx][:, :, :h + 1].clone()
    y[h], y[:, h], y[:, :, h] = 0.0, 0.0, 0.0
    return y


def _exact_gradient(case, seed):
    n, box, kb, nb = case["n"], case["box"], _kbins(case), case["nbins"]
    d, _, _ = _pair(case, seed, case["n_gal"], 0)
    pos = d.pos.detach()
    gp, gb = _cotangents(case, seed)
    ng, vol = case["n_gal"], box**3
    i22, n0, i33 = ng * ng / vol, vol / ng, ng**3 / vol**2
    mesh = torch.zeros((n,) * 3, device=DEV, dtype=torch.float64)
    _paint(mesh, pos, torch.ones(ng, device=DEV, dtype=torch.float64), n, box, (0.0, 0.0, 0.0), 3, 0.0)
    x = torch.fft.rfftn(mesh - ng / float(n) ** 3)
    del mesh
    # every binned mode and every product of two or three of them fits a grid of m points per side
    kmax = kb[0] + nb * kb[1]
    m = min(n, 2 * (int(2 * kmax * box / (2 * math.pi)) + 2))
    x = _coarse(x, n, m) if m < n else x
    i, j, l_ = _modes(m)
    win = 1.0
    for a in (i, j, l_):
        win = win * torch.sinc(a / n) ** 3
    x = x / win
    b, _, wt = _bins(m, box, kb)
    cnt = _binsum(wt, b, nb)
    div = cnt.clamp_min(1.0)
    mu = _mu_z(m)
    p, kern = [], torch.zeros_like(wt)
    for e, l in enumerate((0, 2, 4)):
        lmu = _legendre(l, mu).expand_as(wt)
        p.append((2 * l + 1) / i22 * _binsum(wt * lmu * (x.real**2 + x.imag**2), b, nb) / div - (n0 if l == 0 else 0.0))
        coef = torch.cat([torch.zeros(1, device=DEV, dtype=torch.float64), (2 * l + 1) / i22 * gp[e] / div])
        kern += lmu * coef[b + 1]
    gx = 2.0 * kern * x
    b0, nts = [], []
    for q in range(nb):
        f = _real(torch.where(b == q, x, 0.0), m)
        nt = (_real((b == q).to(x.dtype), m) ** 3).sum() / float(m) ** 3
        b0.append((f**3).sum() / float(m) ** 3 / (i33 * nt))
        nts.append(torch.round(nt))
        # d B0 / d X: 3 F^2 transformed back, sums over the fine grid being (n/m)^3 those over this one
        dq = torch.fft.rfftn(f * f) / float(m) ** 3
        gx += torch.where(b == q, 3.0 * gb[q] / (i33 * nt) * dq, 0.0)
    gx = gx / win
    if m < n:
        h = m // 2
        idx = torch.tensor(list(range(h)) + list(range(n - h + 1, n)), device=DEV)
        src = torch.tensor(list(range(h)) + list(range(h + 1, m)), device=DEV)
        full = torch.zeros((n, n, n // 2 + 1), device=DEV, dtype=x.dtype)
        full[idx[:, None], idx[None, :], :h] = gx[src[:, None], src[None, :], :h]
        gx = full
    gm = _real(gx, n).reshape(-1)
    del gx
    grads = []
    for pc in pos.split(1 << 21):
        i0, taps = _taps(pc.double() * (n / box), 3)
        acc = torch.zeros((len(pc), 3), device=DEV, dtype=torch.float64)
        for ox, wx, dx in taps:
            for oy, wy, dy in taps:
                ixy = ((i0[:, 0] + ox) % n * n + (i0[:, 1] + oy) % n) * n
                for oz, wz, dz in taps:
                    v = gm[ixy + (i0[:, 2] + oz) % n]
                    acc[:, 0] += v * dx[:, 0] * wy[:, 1] * wz[:, 2]
                    acc[:, 1] += v * wx[:, 0] * dy[:, 1] * wz[:, 2]
                    acc[:, 2] += v * wx[:, 0] * wy[:, 1] * dz[:, 2]
        grads.append(acc * (n / box))
    return {"P": torch.stack(p), "B0": torch.stack(b0), "NT": torch.stack(nts), "grad": torch.cat(grads)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "power":
        d, r, o = _pair(case, seed, case["n_gal"], case["n_ran"])
        return _exact_power(d, r, case, o, _ints(case["ells"]), _ints(case["modified"]))
    if kind == "cross":
        return _exact_cross(case, seed)
    if kind == "bispec":
        d, r, o = _pair(case, seed, case["n_gal"], case["n_ran"])
        return _exact_bispec(d, r, case, o)
    if kind == "tripo":
        return _exact_tripo(case, seed)
    if kind == "gradient":
        return _exact_gradient(case, seed)
    flat = []
    for it in _batch_items(case, seed):
        base = dict(n=it["n"], box=it["box"], assign=3, interlace=1)
        kmin, dk, nb = it["power_bins"]
        p = _exact_power(it["data"], it["randoms"], dict(base, kmin=kmin, dk=dk, nbins=nb), it["origin"], (0, 2, 4), ())
        kmin, dk, nb = it["bispec_bins"]
        b = _exact_bispec(it["data"], it["randoms"],
                          dict(base, kmin=kmin, dk=dk, nbins=nb, scoc="0", tripo="", shot="analytic"), it["origin"])
        flat += [*p.values(), *b.values()]
    return {"out": torch.cat([v.reshape(-1) for v in flat])}
