"""The workloads whose speed matters to a user of this library, as calls of its public entry points.

A case is one call that a survey analysis makes many times: the ideal power spectrum and bispectrum of a simulation
box (one field a call, or a batch of boxes), the bispectrum multipoles, the numerators of the masked estimators (one
per mock catalogue) and single Monte Carlo terms of their Fisher matrices (tens to hundreds per survey geometry).  The
grids, bins, boxes and masks are those of ``paper_2404_07249_gb300.synth.WORKLOADS`` and of the tests, or smaller and
ragged forms of them.  (The conjugate-gradient weighting is left out: its ten single-precision iterations magnify a
rounding difference to a percent, so two correct results cannot be compared.)

Outputs.  The library hands every host result out as float64, whatever the precision of its arithmetic.  ``run`` keeps
float64 for the double-precision contexts and stores the results of the single-precision ones ("fp32", "split") as
float32, the precision they are computed with.
"""
import math

import numpy as np
import torch

import paper_2404_07249_gb300 as polybin

# ------------------------------------------------------------------------------------------------------ the cases


def listed():
    w512 = 0.01 * 2000.0 / (2.0 * math.pi)          # bins of 0.01 h/Mpc in units of k_F, box 2000 Mpc/h
    return [
        # The smallest call: P_0, P_2, P_4 of a 64^3 box in double precision, a convergence test or a tiny mock.
        dict(name="pk_64_fp64", kind="pk", n0=64, n1=64, n2=64, box=1000.0, first=0.0, width=2.0, nb=16, lmax=4,
             prec="fp64", field="grf", batch=1),
        # The bispectrum of the same box in double precision: the reference path at its usual size.
        dict(name="bk_64_fp64", kind="bkpk", n0=64, n1=64, n2=64, box=1000.0, first=1.0, width=2.0, nb=8, lmax=-1,
             prec="fp64", field="grf", batch=1),
        # P_0, P_2 of a mid-size redshift-space box: what is run on every snapshot, single precision.
        dict(name="pk_256_fp32", kind="pk", n0=256, n1=256, n2=256, box=2000.0, first=0.0, width=w512, nb=20, lmax=2,
             prec="fp32", field="lognormal_kaiser", batch=1),
        # Both statistics of two boxes on an uneven 2-3-5 grid, plain single precision (no tensor cores).
        dict(name="bkpk_150x180x216_fp32", kind="bkpk", n0=150, n1=180, n2=216, box=1500.0, first=0.0, width=2.5,
             nb=13, lmax=2, prec="fp32", field="lognormal", batch=2),
        # The bispectrum of a mid-size lognormal mock: the ordinary covariance-mock call.
        dict(name="bk_256_split", kind="bkpk", n0=256, n1=256, n2=256, box=2000.0, first=0.0, width=w512, nb=20,
             lmax=-1, prec="split", field="lognormal", batch=1),
        # Both statistics of a full-size redshift-space box: the headline workload.
        dict(name="bkpk_512_split", kind="bkpk", n0=512, n1=512, n2=512, box=2000.0, first=0.0, width=w512, nb=30,
             lmax=2, prec="split", field="lognormal_kaiser", batch=1),
        # A batch of 64 small boxes on uneven grids in one call: emulator training sets.
        dict(name="multi_64_split", kind="multi", ga=96, gb=128, gc=160, box=1000.0, first=1.0, width=2.0, nb=12,
             prec="split", field="lognormal", fields=64),
        # B_0, B_2, B_4 of one redshift-space field.
        dict(name="multipoles_256_split", kind="multipoles", n0=256, n1=256, n2=256, box=2000.0, first=0.0,
             width=w512, nb=20, lmax_b=4, prec="split", field="lognormal_kaiser"),
        # Numerator of the masked bispectrum of one catalogue, with the linear term from two mocks.
        dict(name="bk_masked_256_split", kind="bk_masked", n0=256, n1=256, n2=256, box=2500.0, first=1.0, width=2.0,
             nb=16, prec="split", mocks=2),
        # One Monte Carlo term of the masked power spectrum's Fisher matrix, 3 x 24 bins.
        dict(name="pk_fisher_256_split", kind="pk_fisher", n0=256, n1=256, n2=256, box=2500.0, first=0.0, width=2.0,
             nb=24, lmax=4, prec="split"),
        # One Monte Carlo term of the masked bispectrum's Fisher matrix, 564 triplets: the largest single call.
        dict(name="bk_fisher_256_split", kind="bk_fisher", n0=256, n1=256, n2=256, box=2500.0, first=1.0, width=2.0,
             nb=16, prec="split"),
        # Numerator of the masked power spectrum multipoles with a local line of sight (Yamamoto).
        dict(name="pk_local_256_fp32", kind="pk_local", n0=256, n1=256, n2=256, box=2500.0, first=0.0, width=2.0,
             nb=24, lmax=4, prec="fp32"),
    ]


def _smooth(lo, hi):
    out = []
    for n in range(lo + lo % 2, hi + 1, 2):
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1:
            out.append(n)
    return out


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _grid(rng, lo, hi, ragged=True):
    """Three even 2-3-5 lengths in [lo, hi], alike to about 20 percent, spread over the range's logarithm."""
    mid = _log(rng, lo, hi)
    near = [n for n in _smooth(lo, hi) if 0.83 * mid <= n <= 1.2 * mid] or [min(_smooth(lo, hi), key=lambda n: abs(n - mid))]
    if ragged and rng.random() < 0.6:
        return [rng.choice(near) for _ in range(3)]
    return [rng.choice(near)] * 3


def _bins(rng, n, nb_lo, nb_hi, reach=0.96, starts=(0.0, 0.5, 1.0)):
    """First edge, width and number of bins (k_F units) that end below the Nyquist wave number of n points.  (With a
    first edge of 1/2 some triplets are closed by a dozen triangles and their estimate, a sum that cancels to its last
    digits over the count, outweighs all others: the normalised bispectra start their bins at 0 or 1.)"""
    nb = rng.randint(nb_lo, nb_hi)
    first = rng.choice(starts)
    top = (n // 2) * rng.uniform(0.45, reach)
    width = max(1.25 if first == 0.0 else 1.0, round((top - first) / nb * 4.0) / 4.0)   # no bin without modes
    while first + width * nb > n // 2 * reach and nb > 3:
        nb -= 1
    return first, width, nb


def draw(rng):
    kind = rng.choice(["pk", "bkpk", "bkpk", "multi", "multipoles", "bk_masked", "pk_fisher", "bk_fisher", "pk_local"])
    box = rng.choice([1000.0, 1500.0, 2000.0, 2500.0])
    if kind == "pk":
        prec = rng.choice(["fp64", "fp32"])
        g = _grid(rng, 40, 128 if prec == "fp64" else 320)
        first, width, nb = _bins(rng, min(g), 6, 30)
        return dict(kind=kind, n0=g[0], n1=g[1], n2=g[2], box=box, first=first, width=width, nb=nb,
                    lmax=rng.choice([0, 2, 4]), prec=prec, field=rng.choice(["grf", "lognormal_kaiser"]),
                    batch=rng.randint(1, 2))
    if kind == "bkpk":
        prec = rng.choice(["split", "split", "split", "fp32", "fp64"])
        g = _grid(rng, 48, {"split": 480, "fp32": 240, "fp64": 72}[prec])
        first, width, nb = _bins(rng, min(g), 5, 28 if prec == "split" else 12, 0.7, (0.0, 1.0))
        return dict(kind=kind, n0=g[0], n1=g[1], n2=g[2], box=box, first=first, width=width, nb=nb,
                    lmax=rng.choice([-1, 2]), prec=prec, field=rng.choice(["grf", "lognormal", "lognormal_kaiser"]),
                    batch=rng.randint(1, 2) if max(g) < 256 else 1)
    if kind == "multi":
        g = sorted(rng.sample(_smooth(72, 160), 3))
        return dict(kind=kind, ga=g[0], gb=g[1], gc=g[2], box=box, first=1.0, width=2.0,
                    nb=rng.randint(6, min(12, (g[0] // 2 - 3) // 2)), prec="split", field="lognormal",
                    fields=rng.randint(8, 64))
    if kind == "multipoles":
        g = _grid(rng, 64, 270)
        first, width, nb = _bins(rng, min(g), 5, 20, 0.6, (0.0, 1.0))
        return dict(kind=kind, n0=g[0], n1=g[1], n2=g[2], box=box, first=first, width=width, nb=nb,
                    lmax_b=rng.choice([2, 4]), prec=rng.choice(["split", "split", "fp32"]), field="lognormal_kaiser")
    g = _grid(rng, 64, 240 if kind == "bk_fisher" else 270)
    if kind == "pk_fisher":
        first, width, nb = _bins(rng, min(g), 6, 24, 0.5)
        return dict(kind=kind, n0=g[0], n1=g[1], n2=g[2], box=box, first=first, width=width, nb=nb,
                    lmax=rng.choice([0, 2, 4]), prec=rng.choice(["split", "fp32"]))
    if kind == "pk_local":
        first, width, nb = _bins(rng, min(g), 6, 24, 0.5)
        return dict(kind=kind, n0=g[0], n1=g[1], n2=g[2], box=box, first=first, width=width, nb=nb,
                    lmax=rng.choice([2, 4]), prec=rng.choice(["split", "fp32"]))
    first, width, nb = _bins(rng, min(g), 4, 14, 0.3)
    out = dict(kind=kind, n0=g[0], n1=g[1], n2=g[2], box=box, first=first, width=width, nb=nb,
               prec=rng.choice(["split", "split", "fp32"]) if kind == "bk_masked" else "split")
    if kind == "bk_masked":
        out["mocks"] = rng.randint(0, 3)
    return out


def _edges(case):
    kf = 2.0 * math.pi / case["box"]
    return kf * (case["first"] + case["width"] * np.arange(case["nb"] + 1))


def _shape(case):
    return (case["n0"], case["n1"], case["n2"])


# ------------------------------------------------------------------------------------------------------ the inputs


def _kmodes(grid):
    """Integer wave numbers of the rfftn half spectrum (broadcastable) and |n|^2."""
    n = [torch.fft.fftfreq(m, d=1.0 / m, dtype=torch.float64, device="cuda").round() for m in grid[:2]]
    nx, ny = n[0][:, None, None], n[1][None, :, None]
    nz = torch.arange(grid[2] // 2 + 1, dtype=torch.float64, device="cuda")[None, None, :]
    return nx, ny, nz, nx * nx + ny * ny + nz * nz


def _field(grid, box, kind, gen, kmax=None):
    """A Gaussian field with P(k) = 2e4 (k / 0.1)^-1.5, its lognormal transform, and the Kaiser factor 1 + mu^2 / 2."""
    white = torch.randn(grid, generator=gen, device="cuda", dtype=torch.float32)
    spec = torch.fft.rfftn(white)
    del white
    nx, ny, nz, s = _kmodes(grid)
    s[0, 0, 0] = 1.0
    k = (2.0 * math.pi / box) * s.sqrt()
    amp = (2.0e4 * (k / 0.1) ** -1.5 * (float(np.prod(grid)) / box ** 3)).sqrt()
    if kmax is not None:
        amp[k >= kmax] = 0.0
    amp[0, 0, 0] = 0.0
    spec *= amp.float()
    del amp, k
    f = torch.fft.irfftn(spec, s=grid)
    if kind.startswith("lognormal"):
        f = f.exp_()
        f /= f.double().mean()
        f -= 1.0
        if kind == "lognormal_kaiser":
            spec = torch.fft.rfftn(f)
            spec *= (1.0 + 0.5 * (nz * nz / s)).float()
            spec[0, 0, 0] = 0.0
            f = torch.fft.irfftn(spec, s=grid)
    return f.contiguous()


def _mask(grid, box, gen):
    """Background density of a survey shell around the box centre with 20 holes (synth.SurveyGeometry scaled to the
    box)."""
    u = box / 2500.0
    r_min, r_max, hole = 600.0 * u, 1400.0 * u, 50.0 * u
    q = torch.rand(20, generator=gen, device="cuda", dtype=torch.float64)
    v = torch.randn((20, 3), generator=gen, device="cuda", dtype=torch.float64)
    c = (v / v.norm(dim=1, keepdim=True) * ((r_min ** 3 + q * (r_max ** 3 - r_min ** 3)) ** (1.0 / 3.0))[:, None]).tolist()
    x, y, z = _cells(grid, box)
    r2 = x * x + y * y + z * z
    r = r2.sqrt()
    inside = (r > r_min) & (r < r_max)
    for cx, cy, cz in c:
        inside &= r2 - 2.0 * (cx * x + cy * y + cz * z) + (cx * cx + cy * cy + cz * cz) >= hole * hole
    n = 3.0e-4 * torch.exp(-((r / u - 1000.0) ** 2) / 4.0e5)
    return torch.where(inside, n, torch.zeros_like(n)).float().contiguous()


def _cells(grid, box):
    ax = [(torch.arange(m, dtype=torch.float64, device="cuda") + 0.5) * (box / m) - box / 2.0 for m in grid]
    return ax[0][:, None, None], ax[1][None, :, None], ax[2][None, None, :]


P_FKP = 1.0e4


def _inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    kind = case["kind"]
    if kind == "multi":
        grids = [(case[g],) * 3 for g in ("ga", "gb", "gc")]
        order = [grids[i % 3] for i in range(case["fields"])]
        return {"order": order, "fields": [_field(g, case["box"], case["field"], gen) for g in order]}
    grid, box = _shape(case), case["box"]
    if kind in ("pk", "bkpk"):
        f = [_field(grid, box, case["field"], gen) for _ in range(case["batch"])]
        return {"delta": torch.stack(f) if len(f) > 1 else f[0]}
    if kind == "multipoles":
        return {"delta": _field(grid, box, case["field"], gen)}
    n = _mask(grid, box, gen)
    if kind in ("pk_fisher", "bk_fisher"):
        return {"n": n}
    kmax = float(_edges(case)[-1])
    d = n * _field(grid, box, "grf", gen, kmax)
    out = {"n": n, "d": d, "mocks": None}
    if case.get("mocks"):
        out["mocks"] = torch.stack([n * _field(grid, box, "grf", gen, kmax) for _ in range(case["mocks"])])
    return out


def prepare(case, seed):
    """The fields and masks, the context of the grid and bins with its mode counts, and for the masked estimators the
    FKP weights: made once per geometry by a user's program."""
    state = _inputs(case, seed)
    state["case"] = case
    state["seed"] = int(seed)
    edges = _edges(case)
    if case["kind"] == "multi":
        pbs = {g: polybin.PolyBin(g, case["box"], edges, prec=case["prec"]) for g in set(state["order"])}
        for pb in pbs.values():
            pb.num_triplets()
        state["pbs"] = [pbs[g] for g in state["order"]]
        return state
    pb = polybin.PolyBin(_shape(case), case["box"], edges, lmax=max(0, case.get("lmax", 0)), prec=case["prec"])
    if case["kind"] in ("bkpk", "multipoles", "bk_masked", "bk_fisher"):
        pb.num_triplets()
    if case["kind"] == "pk_local":
        pb.set_observer((0.0, 0.0, 0.0))
    if "n" in state:
        state["w"] = pb.fkp_weights(state["n"], P_FKP)
    state["pb"] = pb
    return state


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "multi":
        out = {"B": polybin.bk_ideal_multi(state["pbs"], state["fields"])}
    elif kind == "pk":
        out = {"P": state["pb"].pk(state["delta"])}
    elif kind == "bkpk":
        if case["lmax"] >= 0:
            B, P = state["pb"].bk_pk(state["delta"])
            out = {"B": B, "P": P}
        else:
            out = {"B": state["pb"].bk_ideal(state["delta"])}
    elif kind == "multipoles":
        out = {"B": state["pb"].bk_multipoles(state["delta"], case["lmax_b"])}
    elif kind == "bk_masked":
        _, num, lin = state["pb"].bk_unwindowed(state["d"], state["w"], state["mocks"], with_estimate=False)
        out = {"num": num, "lin": lin}
    elif kind == "pk_local":
        out = {"num": state["pb"].pk_unwindowed_local(state["d"], state["w"], with_estimate=False)[1]}
    else:
        which = polybin.FISHER_PK if kind == "pk_fisher" else polybin.FISHER_BK
        out = {"F": state["pb"].fisher_draws(state["n"], state["w"], state["seed"], which, 0, 1)}
    return _as_computed(out, case["prec"])


def _as_computed(out, prec):
    """Single-precision results as float32: the trailing digits of their float64 form hold no more."""
    if prec == "fp64":
        return out
    return {k: [x.astype(np.float32) for x in v] if isinstance(v, list) else v.astype(np.float32) for k, v in out.items()}


# ------------------------------------------------------------------------------------------------------ the work


def _closed(case):
    """Number of bin triplets a <= b <= c that hold triangles, by their edges."""
    e = [case["first"] + case["width"] * i for i in range(case["nb"] + 1)]
    nb = case["nb"]
    return sum(1 for a in range(nb) for b in range(a, nb) for c in range(b, nb) if e[a + 1] + e[b + 1] > e[c])


def _cells_needed(case, grid):
    """Cells of the smallest alias-free grid of a triple sum (more than 3 m points an axis, at most the data's)."""
    m = case["first"] + case["width"] * case["nb"]
    return float(np.prod([min(g, 3.0 * min(m, g / 2.0) + 1.0) for g in grid]))


def _fft_flops(n):
    return 2.5 * n * math.log2(n)                    # a real transform of n points


def work(case):
    """Each field read once, the results written once; real transforms at 5/2 n log2 n and two operations for each
    closed triplet on each cell of the alias-free grid."""
    kind = case["kind"]
    nt = _closed(case) if kind not in ("pk", "pk_fisher", "pk_local") else 0
    if kind == "multi":
        total = {"bytes": 0.0, "flops": 0.0}
        for i in range(case["fields"]):
            g = (case[("ga", "gb", "gc")[i % 3]],) * 3
            n, c = float(np.prod(g)), _cells_needed(case, g)
            total["bytes"] += 4.0 * n + 8.0 * nt
            total["flops"] += _fft_flops(n) + case["nb"] * _fft_flops(c) + 2.0 * nt * c
        return total
    grid = _shape(case)
    n, c = float(np.prod(grid)), _cells_needed(case, grid)
    nb = case["nb"]
    if kind in ("pk", "bkpk"):
        nl = case["lmax"] // 2 + 1 if case["lmax"] >= 0 else 0
        f = _fft_flops(n) + (nb * _fft_flops(c) + 2.0 * nt * c if kind == "bkpk" else 0.0)
        return {"bytes": case["batch"] * (4.0 * n + 8.0 * (nt + nl * nb)), "flops": case["batch"] * f}
    if kind == "multipoles":
        nl = case["lmax_b"] // 2 + 1
        return {"bytes": 4.0 * n + 8.0 * nl * nt, "flops": _fft_flops(n) + nl * (nb * _fft_flops(c) + 2.0 * nt * c)}
    if kind == "bk_masked":
        k = case["mocks"]
        return {"bytes": 4.0 * n * (2 + k) + 16.0 * nt,
                "flops": (1 + k) * (_fft_flops(n) + nb * _fft_flops(c)) + (1 + 3 * k) * 2.0 * nt * c}
    if kind == "pk_local":
        forms = sum(2 * ell + 1 for ell in range(0, case["lmax"] + 1, 2))
        return {"bytes": 8.0 * n + 8.0 * nb * (case["lmax"] // 2 + 1), "flops": forms * _fft_flops(n)}
    if kind == "pk_fisher":
        na = (case["lmax"] // 2 + 1) * nb
        return {"bytes": 8.0 * n + 8.0 * na * na, "flops": (2 + 2 * na) * _fft_flops(n)}
    pairs = nb * (nb + 1) // 2
    modes = 2.0 / 3.0 * math.pi * (case["first"] + case["width"] * nb) ** 3
    return {"bytes": 8.0 * n + 8.0 * nt * nt,
            "flops": 4.0 * (_fft_flops(n) + (nb + pairs) * _fft_flops(c)) + 2.0 * nt * _fft_flops(n) +
            4.0 * nt * nt * modes}


# ------------------------------------------------------------------------------------------------------ in 64 bits


def _bin_index(case, s):
    """Bin of each mode of the half spectrum from the integer |n|^2; -1 outside."""
    edges = torch.from_numpy(_edges(case)).cuda()
    k = (2.0 * math.pi / case["box"]) * s.sqrt()
    b = torch.bucketize(k, edges, right=True) - 1
    return torch.where((s > 0) & (b >= 0) & (b < case["nb"]), b, torch.full_like(b, -1))


def _half_weight(grid):
    """How often a mode of the half spectrum stands in the full one."""
    w = torch.full((grid[2] // 2 + 1,), 2.0, dtype=torch.float64, device="cuda")
    w[0] = 1.0
    w[-1] = 1.0
    return w[None, None, :].expand(grid[0], grid[1], -1)


def _legendre(ell, mu2):
    if ell == 0:
        return torch.ones_like(mu2)
    return 0.5 * (3.0 * mu2 - 1.0) if ell == 2 else (35.0 * mu2 * mu2 - 30.0 * mu2 + 3.0) / 8.0


def _shells(spec, bins, nb, grid):
    out = torch.empty((nb, int(np.prod(grid))), dtype=torch.float64, device="cuda")
    zero = torch.zeros((), dtype=spec.dtype, device="cuda")
    for b in range(nb):
        out[b] = torch.fft.irfftn(torch.where(bins == b, spec, zero), s=grid).reshape(-1)
    return out


def _triple(x, y, z, ordered=True):
    """sum over cells of x_a y_b z_c for all a, b, c (``ordered``: b, c >= a only)."""
    nb, n = x.shape
    out = torch.zeros((nb, nb, nb), dtype=torch.float64, device="cuda")
    step = 1 << 22
    for i in range(0, n, step):
        xs, ys, zs = x[:, i:i + step], y[:, i:i + step], z[:, i:i + step]
        for a in range(nb):
            lo = a if ordered else 0
            out[a, lo:, lo:] += (ys[lo:] * xs[a]) @ zs[lo:].T
    return out


def _triplets(case, grid):
    """The closed triplets and T_abc = sum over cells of the unit shells' product, N_abc / N^2 by the number N_abc of
    closed triangles; counted on the smallest grid of more than 3 m points an axis, m the largest binned wave number,
    where the data grid has more."""
    nb, n = case["nb"], float(np.prod(grid))
    m = int(case["first"] + case["width"] * nb) + 1
    small = tuple(min(g, 3 * m + 2 + m % 2) for g in grid)
    bins = _bin_index(case, _kmodes(small)[3])
    one = torch.ones(bins.shape, dtype=torch.complex128, device="cuda")
    t = _shells(one, bins, nb, small)
    count = (_triple(t, t, t) * float(np.prod(small)) ** 2).round().cpu().numpy()
    return [(a, b, c) for a in range(nb) for b in range(a, nb) for c in range(b, nb) if count[a, b, c] > 0], count / n ** 2


def _pick(M, trip):
    M = M.cpu().numpy() if isinstance(M, torch.Tensor) else M
    return np.array([M[t] for t in trip])


def _exact_bk(case, delta, grid, trip, T, bins):
    D = torch.fft.rfftn(delta.double())
    g = _shells(D, bins, case["nb"], grid)
    V, n = case["box"] ** 3, float(np.prod(grid))
    return V * V / n ** 3 * _pick(_triple(g, g, g), trip) / _pick(T, trip)


def _exact_pk(case, delta, grid, bins, s, nz):
    D = torch.fft.rfftn(delta.double())
    w = _half_weight(grid)
    sel = bins >= 0
    idx, n = bins[sel], float(np.prod(grid))
    pw = ((D.real ** 2 + D.imag ** 2) * w)[sel]
    mu2 = (nz * nz / s.clamp(min=1.0))[sel]
    count = torch.bincount(idx, weights=w[sel], minlength=case["nb"])
    rows = [(2 * ell + 1) * case["box"] ** 3 / n ** 2 *
            torch.bincount(idx, weights=pw * _legendre(ell, mu2), minlength=case["nb"]) / count
            for ell in range(0, case["lmax"] + 1, 2)]
    return torch.stack(rows).cpu().numpy()


def _philox(n, seed, number, stream):
    """Flat white noise of the library's Monte Carlo draws (Philox4x32-10, counter (j, 0, number, stream), Box-Muller),
    rounded to float32 as the single-precision contexts define them."""
    m32 = 0xFFFFFFFF
    j = torch.arange((n + 3) // 4, dtype=torch.int64, device="cuda")
    c = [j & m32, j >> 32, torch.full_like(j, number), torch.full_like(j, stream)]
    k0, k1 = seed & m32, (seed >> 32) & m32

    def mul(a, m):                                   # high and low words of a 32 x 32 bit product, in 16-bit halves
        lo = a * (m & 0xFFFF)
        hi = a * (m >> 16) + (lo >> 16)
        return hi >> 16, ((hi & 0xFFFF) << 16) | (lo & 0xFFFF)

    for _ in range(10):
        h0, l0 = mul(c[0], 0xD2511F53)
        h1, l1 = mul(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    u = [(x.double() + 0.5) * 2.0 ** -32 for x in c]
    r0, r1 = (-2.0 * u[0].log()).sqrt(), (-2.0 * u[2].log()).sqrt()
    z = torch.stack([r0 * torch.cos(2.0 * math.pi * u[1]), r0 * torch.sin(2.0 * math.pi * u[1]),
                     r1 * torch.cos(2.0 * math.pi * u[3]), r1 * torch.sin(2.0 * math.pi * u[3])], dim=1)
    return z.reshape(-1)[:n].float().double()


def _exact_pk_fisher(case, n, w, seed, grid, bins, s, nz):
    N = int(np.prod(grid))
    a = _philox(N, seed, 0, 2).reshape(grid)
    sw = w * n
    A, SA = torch.fft.rfftn(a), torch.fft.rfftn(sw * a)
    sel, mu2 = bins >= 0, nz * nz / s.clamp(min=1.0)
    hw = _half_weight(grid)[sel]
    alphas = [(ell, b) for ell in range(0, case["lmax"] + 1, 2) for b in range(case["nb"])]
    L = {ell: _legendre(ell, mu2) for ell, _ in alphas}
    idx = bins[sel]
    Y = torch.stack([torch.where(idx == b, L[ell][sel] * A[sel], 0.0 * A[sel]) for ell, b in alphas])
    X = torch.stack([torch.fft.rfftn(sw * torch.fft.irfftn(torch.where(bins == b, L[ell] * SA, 0.0 * SA), s=grid))[sel]
                     for ell, b in alphas])
    return (0.5 / N * ((X.conj() * hw) @ Y.T).real).cpu().numpy()[None]


def _exact_bk_fisher(case, n, w, seed, grid, bins, trip):
    N, nb = int(np.prod(grid)), case["nb"]
    sw = w * n
    sel = bins >= 0
    idx, hw = bins[sel], _half_weight(grid)[sel]
    pairs = [(i, j) for i in range(nb) for j in range(i, nb)]

    def pair_differences(scale):
        """FT[g_i g_j] on the binned modes, the first draw's minus the second's."""
        out = {}
        for stream, sign in ((0, 1.0), (1, -1.0)):
            a = _philox(N, seed, 0, stream).reshape(grid)
            g = _shells(torch.fft.rfftn(a * scale if scale is not None else a), bins, nb, grid)
            for i, j in pairs:
                f = sign * torch.fft.rfftn((g[i] * g[j]).reshape(grid))[sel]
                out[i, j] = out[i, j] + f if (i, j) in out else f
        return out

    at = [idx == b for b in range(nb)]

    def q(P, a, b, c):
        delta = 6.0 if a == b == c else 2.0 if a == b or b == c else 1.0
        return 2.0 / delta * (at[c] * P[a, b] + at[a] * P[b, c] + at[b] * P[a, c])

    PX = pair_differences(sw)
    X = torch.empty((len(trip), idx.numel()), dtype=torch.complex128, device="cuda")
    spec = torch.zeros(bins.shape, dtype=torch.complex128, device="cuda")
    for t, (a, b, c) in enumerate(trip):
        spec[sel] = q(PX, a, b, c)
        X[t] = torch.fft.rfftn(sw * torch.fft.irfftn(spec, s=grid))[sel]
    del PX
    PY = pair_differences(None)
    X = X.conj() * hw
    F = torch.empty((len(trip), len(trip)), dtype=torch.float64, device="cuda")
    for t0 in range(0, len(trip), 64):
        Y = torch.stack([q(PY, *t) for t in trip[t0:t0 + 64]])
        F[:, t0:t0 + 64] = (X @ Y.T).real
    return (F / (24.0 * N)).cpu().numpy()[None]


def _exact_pk_local(case, d, w, grid, bins, modes):
    """sum_m Ybar_lm(k) FT[Ybar_lm(x) u] = FT_x[L_l(k.x) u], by the monomials of the Legendre polynomials."""
    u = d * w
    N = float(np.prod(grid))
    x, y, z = _cells(grid, case["box"])
    r = (x * x + y * y + z * z).sqrt()
    xh = [c / r for c in (x, y, z)]
    nx, ny, nz, s = modes
    kr = s.clamp(min=1.0).sqrt()
    kh = [c / kr for c in (nx, ny, nz)]

    def power(p):
        """FT_x[(k.x)^p u]."""
        out = 0.0
        for i in range(p + 1):
            for j in range(p + 1 - i):
                l = p - i - j
                m = math.factorial(p) // (math.factorial(i) * math.factorial(j) * math.factorial(l))
                out = out + m * kh[0] ** i * kh[1] ** j * kh[2] ** l * \
                    torch.fft.rfftn(xh[0] ** i * xh[1] ** j * xh[2] ** l * u)
        return out

    U = torch.fft.rfftn(u)
    q = {0: U}
    if case["lmax"] >= 2:
        q[2] = power(2)
    if case["lmax"] >= 4:
        q[4] = power(4)
    sel = bins >= 0
    hw = _half_weight(grid)
    rows = []
    for ell in range(0, case["lmax"] + 1, 2):
        A = U if ell == 0 else 0.5 * (3.0 * q[2] - U) if ell == 2 else (35.0 * q[4] - 30.0 * q[2] + 3.0 * U) / 8.0
        v = ((A.conj() * U).real * hw)[sel]
        rows.append(0.5 / N * torch.bincount(bins[sel], weights=v, minlength=case["nb"]))
    return torch.cat(rows).cpu().numpy()


def exact(case, seed):
    x = _inputs(case, seed)
    kind, nb = case["kind"], case["nb"]
    if kind == "multi":
        plans, out = {}, []
        for g, f in zip(x["order"], x["fields"]):
            if g not in plans:
                bins = _bin_index(case, _kmodes(g)[3])
                plans[g] = (bins,) + _triplets(case, g)
            bins, trip, T = plans[g]
            out.append(_exact_bk(case, f, g, trip, T, bins))
        return {"B": out}
    grid = _shape(case)
    modes = _kmodes(grid)
    nz, s = modes[2], modes[3]
    bins = _bin_index(case, s)
    if kind in ("pk", "bkpk"):
        fields = x["delta"] if x["delta"].ndim == 4 else x["delta"][None]
        out = {}
        if kind == "bkpk":
            trip, T = _triplets(case, grid)
            out["B"] = np.stack([_exact_bk(case, f, grid, trip, T, bins) for f in fields])
        if case["lmax"] >= 0:
            out["P"] = np.stack([_exact_pk(case, f, grid, bins, s, nz) for f in fields])
        return out
    if kind == "multipoles":
        trip, T = _triplets(case, grid)
        D = torch.fft.rfftn(x["delta"].double())
        g = _shells(D, bins, nb, grid)
        mu2 = nz * nz / s.clamp(min=1.0)
        V, N = case["box"] ** 3, float(np.prod(grid))
        rows = []
        for ell in range(0, case["lmax_b"] + 1, 2):
            h = _shells(D * _legendre(ell, mu2), bins, nb, grid)
            rows.append((2 * ell + 1) * V * V / N ** 3 * _pick(_triple(g, g, h), trip) / _pick(T, trip))
        return {"B": np.stack(rows)[None]}
    n = x["n"].double()
    w = 1.0 / (n * P_FKP + 1.0)
    if kind == "pk_fisher":
        return {"F": _exact_pk_fisher(case, n, w, int(seed), grid, bins, s, nz)}
    if kind == "pk_local":
        return {"num": _exact_pk_local(case, x["d"].double(), w, grid, bins, modes)}
    trip, _ = _triplets(case, grid)
    if kind == "bk_fisher":
        return {"F": _exact_bk_fisher(case, n, w, int(seed), grid, bins, trip)}
    g = _shells(torch.fft.rfftn(w * x["d"].double()), bins, nb, grid)
    S = _pick(_triple(g, g, g), trip)
    lin = np.zeros(len(trip))
    mocks = x["mocks"] if x["mocks"] is not None else []
    for m in mocks:
        h = _shells(torch.fft.rfftn(w * m.double()), bins, nb, grid)
        lin += _pick(_triple(g, h, h, False), trip) + _pick(_triple(h, g, h, False), trip) + \
            _pick(_triple(h, h, g, False), trip)
    lin /= max(1, len(mocks))
    delta = np.array([6.0 if a == b == c else 2.0 if a == b or b == c else 1.0 for a, b, c in trip])
    return {"num": (S - lin) / delta, "lin": lin}
