"""The transforms a user of this library runs, as measurable cases.

Every case goes through the public calls (``sht_execute``, ``sht_batch_execute``,
``autograd.synthesis``) with the plan a program keeps.  Kinds:

  pair      synthesis a_lm -> maps, then weighted analysis of those maps
  adjoint   adjoint synthesis of given maps, then adjoint analysis of the result
            (the two directions an iterative solver alternates between)
  jacobi    weighted analysis of a HEALPix map refined by three residual steps
  deriv     first-derivative synthesis of scalar coefficients (spin-1 plan)
  grad      ||synthesis(a_lm) - d||^2 and its gradient by torch.autograd
  batch     uneven scalar pairs and one multi-map pair in one batched launch per stage

``exact`` evaluates the same transforms in IEEE double with torch operations on
whole arrays (its own grids, recursion and Fourier sums).
"""
import functools
import math

import numpy as np
import torch

from paper_1303_4945_gb300 import autograd, sht

# Gauss-Legendre and Clenshaw-Curtis cases: nlat rings of nlon points; HEALPix: nside.


def listed():
    return [
        # the smallest call: a scalar pair at lmax 127, where launches and latency count
        {"name": "gl127_s0_fp64", "kind": "pair", "grid": "gauss", "lmax": 127, "nlat": 128, "nlon": 255,
         "spin": 0, "ncomp": 1, "precision": "fp64"},
        # a small polarisation map in the mixed form on odd, non-minimal sizes (prime ring length)
        {"name": "gl300_s2_mixed", "kind": "pair", "grid": "gauss", "lmax": 300, "nlat": 311, "nlon": 613,
         "spin": 2, "ncomp": 1, "precision": "mixed"},
        # the two adjoints of an iterative solver on a Clenshaw-Curtis grid, two scalar maps, FP64
        {"name": "cc511_adj_s0_fp64", "kind": "adjoint", "grid": "cc", "lmax": 511, "nlat": 1025, "nlon": 1024,
         "spin": 0, "ncomp": 2, "precision": "fp64"},
        # the derivative synthesis of a scalar field (lensing, gradients)
        {"name": "gl1535_deriv_mixed", "kind": "deriv", "grid": "gauss", "lmax": 1535, "nlat": 1536, "nlon": 3072,
         "spin": 1, "ncomp": 1, "precision": "mixed"},
        # map making's weighted analysis with three refinement steps at Nside 512, mixed
        {"name": "hp512_jacobi_mixed", "kind": "jacobi", "grid": "healpix", "lmax": 1535, "nside": 512,
         "spin": 0, "ncomp": 1, "precision": "mixed"},
        # a polarisation pair on HEALPix Nside 256 in the FP64 form
        {"name": "hp256_s2_fp64", "kind": "pair", "grid": "healpix", "lmax": 767, "nside": 256,
         "spin": 2, "ncomp": 1, "precision": "fp64"},
        # a mid-size scalar pair in the FP64 form
        {"name": "gl1023_s0_fp64", "kind": "pair", "grid": "gauss", "lmax": 1023, "nlat": 1024, "nlon": 2047,
         "spin": 0, "ncomp": 1, "precision": "fp64"},
        # eight scalar maps of one geometry at once (Monte Carlo simulations), mixed
        {"name": "gl2047_s0_8maps_mixed", "kind": "pair", "grid": "gauss", "lmax": 2047, "nlat": 2048, "nlon": 4095,
         "spin": 0, "ncomp": 8, "precision": "mixed"},
        # independent scalar pairs of uneven size in one launch per stage, mixed
        {"name": "batch24_mixed", "kind": "batch", "problems": 24, "lmin": 64, "lmax": 2047, "sizes": 3, "maps": 4,
         "precision": "mixed"},
        # the headline: a polarisation pair at lmax 4095 in the mixed form
        {"name": "gl4095_s2_mixed", "kind": "pair", "grid": "gauss", "lmax": 4095, "nlat": 4096, "nlon": 8191,
         "spin": 2, "ncomp": 1, "precision": "mixed"},
        # the same size scalar pair, one map, mixed
        {"name": "gl4095_s0_mixed", "kind": "pair", "grid": "gauss", "lmax": 4095, "nlat": 4096, "nlon": 8191,
         "spin": 0, "ncomp": 1, "precision": "mixed"},
        # the largest: loss and gradient of a scalar synthesis at lmax 8191, mixed
        {"name": "gl8191_grad_s0_mixed", "kind": "grad", "grid": "gauss", "lmax": 8191, "nlat": 8192, "nlon": 16383,
         "spin": 0, "ncomp": 1, "precision": "mixed"},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pair", "pair", "pair", "adjoint", "jacobi", "deriv", "grad", "batch"])
    prec = rng.choice(["mixed", "mixed", "fp64"])
    top = 4095 if prec == "mixed" else 1023
    if kind == "jacobi":
        nside = _logint(rng, 48, 512 if prec == "mixed" else 256)
        return {"kind": kind, "grid": "healpix", "lmax": rng.randint(2 * nside, 3 * nside - 1), "nside": nside, "spin": 0,
                "ncomp": 1, "precision": prec}
    if kind == "batch":
        return {"kind": kind, "problems": rng.randint(4, 24), "lmin": 64, "lmax": _logint(rng, 256, min(top, 2047)),
                "sizes": rng.randrange(1 << 20), "maps": rng.choice([1, 2, 3, 4]), "precision": prec}
    lmax = _logint(rng, 100, top)
    spin = {"deriv": 1, "grad": rng.choice([0, 2])}.get(kind, rng.choice([0, 0, 1, 2, 2, 3]))
    ncomp = 1 if kind in ("deriv", "grad") or lmax > 2048 else rng.choice([1, 1, 2, 3, 4])
    grid = rng.choice(["gauss", "gauss", "healpix"]) if kind == "pair" else ("cc" if kind == "adjoint" else "gauss")
    if grid == "healpix":
        nside = max(34, -(-lmax // 3) + rng.randint(0, 16))
        return {"kind": kind, "grid": grid, "lmax": lmax, "nside": nside, "spin": spin, "ncomp": ncomp, "precision": prec}
    if grid == "cc":
        nlat, nlon = 2 * lmax + 3, 2 * lmax + 2
    else:
        nlat, nlon = lmax + 1 + rng.randint(0, 9), 2 * lmax + 1 + rng.choice([0, 0, 1, rng.randint(0, 40)])
    return {"kind": kind, "grid": grid, "lmax": lmax, "nlat": nlat, "nlon": nlon, "spin": spin, "ncomp": ncomp,
            "precision": prec}


# ---- inputs (torch only: exact() draws the same ones) ---------------------------------------------------


def _lm(lmax, dev):
    """(l, m) of every stored coefficient (triangular m-major order)."""
    l = torch.arange(lmax + 1, device=dev, dtype=torch.int32).expand(lmax + 1, lmax + 1)
    keep = l >= l.T
    return l[keep].double(), l.T[keep]


def _gaussian_alm(gen, lmax, n, spin):
    """n arrays of Gaussian coefficients with C_l = 1/(l+1)^2, none below l = |spin|."""
    l, m = _lm(lmax, gen.device)
    sd = torch.where(m == 0, 1.0, math.sqrt(0.5)).double() / (l + 1.0) * (l >= spin)
    out = []
    for _ in range(n):
        a = torch.randn(2, l.numel(), dtype=torch.float64, device=gen.device, generator=gen) * sd
        a[1][m == 0] = 0.0
        out.append(torch.complex(a[0], a[1]))
    return out


def _generator(seed):
    return torch.Generator(device="cuda" if torch.cuda.is_available() else "cpu").manual_seed(seed)


def _npix(case):
    return 12 * case["nside"] ** 2 if case["grid"] == "healpix" else case["nlat"] * case["nlon"]


def _inputs(case, seed):
    gen = _generator(seed)
    spin, narr = case["spin"], case["ncomp"] * (2 if case["spin"] else 1)
    if case["kind"] in ("pair", "deriv"):
        n = case["ncomp"] if case["kind"] == "deriv" else narr
        return {"alm": _gaussian_alm(gen, case["lmax"], n, 0 if case["kind"] == "deriv" else spin)}
    if case["kind"] == "jacobi":  # a smooth sky (spectrum 1/(l+1)^2 in the mean) plus pixel noise
        npix = _npix(case)
        smooth = torch.randn(npix // 16 + 2, dtype=torch.float64, device=gen.device, generator=gen)
        return {"maps": [smooth.repeat_interleave(16)[:npix]
                         + 0.1 * torch.randn(npix, dtype=torch.float64, device=gen.device, generator=gen)]}
    if case["kind"] == "adjoint":
        return {"maps": [torch.randn(_npix(case), dtype=torch.float64, device=gen.device, generator=gen)
                         for _ in range(narr)]}
    alm = _gaussian_alm(gen, case["lmax"], narr, spin)
    return {"alm": alm, "data": torch.randn(narr, _npix(case), dtype=torch.float64, device=gen.device, generator=gen)}


def _batch_problems(case):
    """The batch's problems: (lmax, ncomp), log-uniform sizes, and the multi-map one in the middle of the range."""
    rng = np.random.default_rng(case["sizes"])
    sizes = np.rint(np.exp(rng.uniform(math.log(case["lmin"]), math.log(case["lmax"]), case["problems"]))).astype(int)
    return [(int(l), 1) for l in sizes] + [(int(math.sqrt(case["lmin"] * case["lmax"])), case["maps"])]


def _batch_inputs(case, seed):
    gen = _generator(seed)
    return [_gaussian_alm(gen, lmax, n, 0) for lmax, n in _batch_problems(case)]


# ---- prepare and run ------------------------------------------------------------------------------------


@functools.lru_cache(maxsize=64)
def _geometry(grid, *size):  # a program builds its grid once and keeps the handle
    if grid == "healpix":
        return sht.sht_geom_healpix(*size)
    if grid == "cc":
        return sht.sht_geom_ecp(sht.SHT_ECP_CC, *size)
    return sht.sht_geom_gauss(*size)


def _plan(case):
    size = (case["nside"],) if case["grid"] == "healpix" else (case["nlat"], case["nlon"])
    return sht.sht_plan_create(_geometry(case["grid"], *size), sht.sht_alm_create(case["lmax"], case["lmax"]), case["spin"], case["ncomp"],
                               sht.SHT_MIXED if case["precision"] == "mixed" else sht.SHT_FP64)


def _maps(plan):
    return [torch.empty(plan.geom.npix, dtype=torch.float64, device="cuda") for _ in range(plan.narrays)]


def prepare(case, seed):
    if case["kind"] == "batch":
        alm, plans = _batch_inputs(case, seed), []
        for lmax, n in _batch_problems(case):
            plans.append(_plan({"grid": "gauss", "lmax": lmax, "nlat": lmax + 1, "nlon": 2 * lmax + 1, "spin": 0,
                                "ncomp": n, "precision": case["precision"]}))
        return {"kind": "batch", "batch": sht.sht_batch_create(plans), "alm": alm, "maps": [_maps(p) for p in plans],
                "out": [[torch.empty_like(x) for x in a] for a in alm]}
    plan, given = _plan(case), _inputs(case, seed)
    s = {"kind": case["kind"], "plan": plan, **given}
    if case["kind"] not in ("deriv", "grad"):
        plan.autotune(torch.cuda.current_stream())  # as a program that runs many analyses does
    if case["kind"] == "pair":
        s["maps"], s["out"] = _maps(plan), [torch.empty_like(a) for a in given["alm"]]
    elif case["kind"] == "adjoint":
        s["out"] = [torch.empty(plan.alm.size(), dtype=torch.complex128, device="cuda") for _ in range(plan.narrays)]
        s["back"] = _maps(plan)
    elif case["kind"] == "jacobi":
        s["out"] = torch.empty(plan.alm.size(), dtype=torch.complex128, device="cuda")
        s["work"] = torch.empty_like(given["maps"][0])
    elif case["kind"] == "deriv":
        s["maps"] = _maps(plan)
    else:
        s["alm"] = torch.stack(given["alm"]).requires_grad_()
    return s


def run(s):
    stream = torch.cuda.current_stream()
    kind = s["kind"]
    if kind == "batch":
        sht.sht_batch_execute(s["batch"], sht.SHT_SYNTHESIS, s["alm"], s["maps"], 0, stream)
        sht.sht_batch_execute(s["batch"], sht.SHT_ANALYSIS, s["out"], s["maps"], 0, stream)
        return {"maps": s["maps"], "alm": s["out"]}
    plan = s["plan"]
    if kind == "pair":
        sht.sht_execute(plan, sht.SHT_SYNTHESIS, s["alm"], s["maps"], 0, stream)
        sht.sht_execute(plan, sht.SHT_ANALYSIS, s["out"], s["maps"], 0, stream)
        return {"maps": s["maps"], "alm": s["out"]}
    if kind == "adjoint":
        sht.sht_execute(plan, sht.SHT_ADJOINT_SYNTHESIS, s["out"], s["maps"], 0, stream)
        sht.sht_execute(plan, sht.SHT_ADJOINT_ANALYSIS, s["out"], s["back"], 0, stream)
        return {"alm": s["out"], "maps": s["back"]}
    if kind == "jacobi":
        p, a, r = s["maps"][0], s["out"], s["work"]
        sht.sht_execute(plan, sht.SHT_ANALYSIS, [a], [p], 0, stream)
        for _ in range(3):
            sht.sht_execute(plan, sht.SHT_SYNTHESIS, [a], [r], 0, stream)
            torch.sub(p, r, out=r)
            sht.sht_execute(plan, sht.SHT_ANALYSIS, [a], [r], sht.SHT_ADD_OUTPUT, stream)
        return {"alm": a, "residual": r}
    if kind == "deriv":
        sht.sht_execute(plan, sht.SHT_DERIV_SYNTHESIS, s["alm"], s["maps"], 0, stream)
        return {"maps": s["maps"]}
    a = s["alm"]
    a.grad = None
    r = autograd.synthesis(plan, a) - s["data"]
    loss = torch.dot(r.view(-1), r.view(-1))
    loss.backward()
    return {"loss": loss.detach(), "grad": a.grad}


# ---- the work a pass cannot do without -------------------------------------------------------------------


def _one_way(lmax, spin, ncomp, theta, npix, ring):
    """(bytes, flops) of one transform: arrays read or written once; the (m, l, ring pair) steps left by the polar
    cut with two FMAs of recursion per Legendre function and the multiply-adds into (out of) the sums, and the
    real ring FFTs."""
    t = max(100.0, 0.01 * lmax)
    n = 0.0
    for y in np.unique(np.minimum(theta, math.pi - theta)):
        mtop = spin * math.cos(y) + math.sqrt(max(0.0, (t + lmax * math.sin(y)) ** 2 - (spin * math.sin(y)) ** 2))
        m = min(lmax, int(mtop))
        n += (m + 1.0) * (lmax + 1 - spin) - max(0.0, m - spin) * (m - spin + 1.0) / 2
    narr = ncomp * (2 if spin else 1)
    flops = n * ((8 + 16 * ncomp) if spin else (4 + 4 * ncomp)) + narr * 2.5 * npix * math.log2(max(2, ring))
    return narr * (8.0 * (lmax + 1) * (lmax + 2) + 8.0 * npix), flops


def work(case):
    if case["kind"] == "batch":
        w = [_one_way(l, 0, n, np.linspace(0, math.pi, l + 3)[1:-1], (l + 1) * (2 * l + 1), 2 * l + 1)
             for l, n in _batch_problems(case)]
        return {"bytes": 2 * sum(x[0] for x in w), "flops": 2 * sum(x[1] for x in w)}
    nrings = 4 * case["nside"] - 1 if case["grid"] == "healpix" else case["nlat"]
    ring = 4 * case["nside"] if case["grid"] == "healpix" else case["nlon"]
    b, f = _one_way(case["lmax"], case["spin"], case["ncomp"], np.linspace(0, math.pi, nrings + 2)[1:-1], _npix(case),
                    ring)
    if case["kind"] == "deriv":  # one coefficient array in, two maps out
        return {"bytes": b - 8.0 * (case["lmax"] + 1) * (case["lmax"] + 2), "flops": f}
    times = {"jacobi": 7}.get(case["kind"], 2)
    return {"bytes": times * b, "flops": times * f}


# ---- the same in 64 bits, by whole-array operations ------------------------------------------------------


def _gauss(n):
    """Gauss-Legendre colatitudes and weights: Newton's method on P_n(cos t) in t."""
    t = math.pi * (np.arange(1, n + 1) - 0.25) / (n + 0.5)
    for _ in range(6):
        x, s = np.cos(t), np.sin(t)
        p0, p1 = np.ones(n), x.copy()
        for k in range(2, n + 1):
            p0, p1 = p1, x * p1 + (k - 1.0) / k * (x * p1 - p0)
        d = n * (p0 - x * p1) / s  # sin(t) P_n'(x)
        t = t + p1 / d
    return t, 2.0 / d ** 2


def _cc_weights(n):
    """Clenshaw-Curtis weights at theta = k pi / (n - 1)."""
    big = n - 1
    v = np.zeros(big // 2 + 1)
    k = np.arange(big // 2 + 1)
    v[:] = 2.0 / (1.0 - 4.0 * k ** 2)
    b = np.where((k == 0) | (2 * k == big), 0.5, 1.0)
    th = np.arange(n) * math.pi / big
    w = (2.0 / big) * (np.cos(2.0 * np.outer(th, k)) @ (b * v))
    w[0] *= 0.5
    w[-1] *= 0.5
    return th, w


def _rings(case):
    """theta, nphi, phi0 and pixel weight of every ring, rings stored one after another."""
    if case["grid"] == "healpix":
        ns = case["nside"]
        i = np.arange(1, 4 * ns)
        j = np.minimum(i, 4 * ns - i)
        cap = j < ns
        th = np.where(cap, 2 * np.arcsin(j / (ns * math.sqrt(6.0))), np.arccos(np.minimum(1.0, (2 * ns - j) * 2.0 / (3 * ns))))
        th = np.where(i > 2 * ns, math.pi - th, th)
        nphi = np.where(cap, 4 * j, 4 * ns)
        phi0 = np.where(cap, math.pi / (4 * j), np.where((j - ns) % 2 == 0, math.pi / (4 * ns), 0.0))
        return th, nphi, phi0, np.full(4 * ns - 1, math.pi / (3.0 * ns * ns))
    th, w = _gauss(case["nlat"]) if case["grid"] == "gauss" else _cc_weights(case["nlat"])
    n = case["nlon"]
    return th, np.full(len(th), n), np.zeros(len(th)), w * 2 * math.pi / n


def _start(lmax, s, th, dev):
    """Lambda_{l0,m}(theta) at l0 = max(m, |s|) as mantissa * 2^(600 e), for every m and ring."""
    nm, nr = lmax + 1, len(th)
    val, ex = torch.empty(nm, nr, dtype=torch.float64, device=dev), torch.zeros(nm, nr, dtype=torch.float64, device=dev)
    t = torch.from_numpy(th).to(dev)
    c, sn = torch.cos(t / 2), torch.sin(t / 2)
    a = abs(s)
    cur, e = None, torch.zeros_like(t)
    for m in range(nm):
        if m <= a:  # d^a_{-m,s} by its single term (Wigner's sum at l = |s|)
            f = math.sqrt((2 * a + 1) / (4 * math.pi) * math.comb(2 * a, a + m))
            cur = f * (c ** (a - m) * sn ** (a + m) if s >= 0 else (-1) ** (a + m) * c ** (a + m) * sn ** (a - m))
            cur = cur * (-1) ** m
        else:
            cur = -cur * math.sqrt((2 * m + 1) / (2 * m - 1) * (2 * m) * (2 * m - 1) / ((m - a) * (m + a))) * c * sn
            small = (cur.abs() < 2.0 ** -300) & (cur != 0)
            cur = torch.where(small, cur * 2.0 ** 600, cur)
            e = torch.where(small, e - 1, e)
        val[m], ex[m] = cur, e
    return val, ex


def _legendre(lmax, spin, th, dev, visit):
    """Calls visit(l, {s: Lambda[m <= l, ring]}) for l = |spin| .. lmax, s = spin and -spin."""
    nm = lmax + 1
    sets = (spin, -spin) if spin else (0,)
    a = abs(spin)
    x = torch.cos(torch.from_numpy(th).to(dev))
    m = torch.arange(nm, dtype=torch.float64, device=dev)
    first = {s: _start(lmax, s, th, dev) for s in sets}
    cur = {s: torch.zeros(nm, len(th), dtype=torch.float64, device=dev) for s in sets}
    prev = {s: torch.zeros_like(cur[s]) for s in sets}
    ex = {s: torch.zeros_like(cur[s]) for s in sets}

    def root(l):  # sqrt((l^2 - m^2)(l^2 - s^2) / (4 l^2 - 1)) / l
        return torch.sqrt(((l * l - m * m) * (l * l - a * a)).clamp(min=0.0) / (4.0 * l * l - 1.0)) / l

    for l in range(a, lmax + 1):
        for s in sets:
            new = slice(0, l + 1) if l == a else slice(l, l + 1)
            cur[s][new], ex[s][new] = first[s][0][new], first[s][1][new]
            prev[s][new] = 0.0
        n = l + 1
        visit(l, {s: torch.where(ex[s][:n] == 0, cur[s][:n], 0.0) for s in sets})
        if l == lmax:
            break
        up = root(l + 1.0)[:n, None]
        down = root(float(l))[:n, None] if l > a else torch.zeros(n, 1, dtype=torch.float64, device=dev)
        for s in sets:
            sh = (m[:n, None] * s / (l * (l + 1.0))) if l > 0 and s else 0.0
            nxt = ((x + sh) * cur[s][:n] - down * prev[s][:n]) / up
            prev[s][:n], cur[s][:n] = cur[s][:n].clone(), nxt
            if l % 8 == 0:
                big = (cur[s][:n].abs() > 2.0 ** 300) & (ex[s][:n] < 0)
                cur[s][:n] = torch.where(big, cur[s][:n] * 2.0 ** -600, cur[s][:n])
                prev[s][:n] = torch.where(big, prev[s][:n] * 2.0 ** -600, prev[s][:n])
                ex[s][:n] += big


def _index(lmax, l):
    m = np.arange(l + 1, dtype=np.int64)
    return m * (2 * lmax + 1 - m) // 2 + l


def _to_maps(rings, phase):
    """Real maps from F_m per (m, ring)."""
    th, nphi, phi0, _ = rings
    dev, nm = phase.device, phase.shape[0]
    m = torch.arange(nm, device=dev)
    out = []
    for n, lo, hi in _runs(nphi):
        f = phase[:, lo:hi] * torch.polar(torch.ones((), dtype=torch.float64, device=dev),
                                          m[:, None].double() * torch.from_numpy(phi0[lo:hi]).to(dev))
        z = torch.zeros(n, hi - lo, dtype=torch.complex128, device=dev)
        z.index_add_(0, m % n, f)
        z.index_add_(0, (-m[1:]) % n, f[1:].conj())
        out.append((torch.fft.ifft(z, dim=0).real * n).T.reshape(-1))
    return torch.cat(out)


def _from_maps(rings, p, nm, weighted):
    """G_m per (m, ring) of a real map."""
    th, nphi, phi0, w = rings
    dev = p.device
    m = torch.arange(nm, device=dev)
    out, at = [], 0
    for n, lo, hi in _runs(nphi):
        z = torch.fft.fft(p[at:at + n * (hi - lo)].view(hi - lo, n).T, dim=0)[m % n]
        at += n * (hi - lo)
        g = z * torch.polar(torch.ones((), dtype=torch.float64, device=dev),
                            -m[:, None].double() * torch.from_numpy(phi0[lo:hi]).to(dev))
        out.append(g * torch.from_numpy(w[lo:hi]).to(dev) if weighted else g)
    return torch.cat(out, dim=1)


def _runs(nphi):
    lo = 0
    while lo < len(nphi):
        hi = lo
        while hi < len(nphi) and nphi[hi] == nphi[lo]:
            hi += 1
        yield int(nphi[lo]), lo, hi
        lo = hi


def _synthesis(lmax, spin, rings, alm, weighted=False):
    dev, nr = alm[0].device, len(rings[0])
    f = [torch.zeros(lmax + 1, nr, dtype=torch.complex128, device=dev) for _ in alm]

    def visit(l, lam):
        at = torch.from_numpy(_index(lmax, l)).to(dev)
        if not spin:
            for k, a in enumerate(alm):
                f[k][:l + 1] += a[at][:, None] * lam[0]
            return
        sg = (-1) ** spin
        for k in range(0, len(alm), 2):  # Q + iU from sa = -(E + iB), (-s)a = -(-1)^s (E - iB)
            e, b = alm[k][at].clone(), alm[k + 1][at].clone()
            e[0], b[0] = e[0].real + 0j, b[0].real + 0j
            u, v = -(e + 1j * b)[:, None] * lam[spin], -sg * (e - 1j * b)[:, None] * lam[-spin]
            f[k][:l + 1] += 0.5 * (u + v)
            f[k + 1][:l + 1] += -0.5j * (u - v)

    _legendre(lmax, spin, rings[0], dev, visit)
    for x in f:
        x[0] = x[0].real + 0j
    if weighted:
        w = torch.from_numpy(rings[3]).to(dev)
        f = [x * w for x in f]
    return [_to_maps(rings, x) for x in f]


def _analysis(lmax, spin, rings, maps, weighted=True):
    dev = maps[0].device
    g = [_from_maps(rings, p, lmax + 1, weighted) for p in maps]
    out = [torch.zeros((lmax + 1) * (lmax + 2) // 2, dtype=torch.complex128, device=dev) for _ in maps]

    def visit(l, lam):
        at = torch.from_numpy(_index(lmax, l)).to(dev)

        def dot(z, t):
            z = z[:l + 1]
            return torch.complex((z.real * t).sum(1), (z.imag * t).sum(1))

        if not spin:
            for k in range(len(maps)):
                out[k][at] = dot(g[k], lam[0])
            return
        sg = (-1) ** spin
        for k in range(0, len(maps), 2):
            u, v = dot(g[k] + 1j * g[k + 1], lam[spin]), dot(g[k] - 1j * g[k + 1], lam[-spin])
            out[k][at] = -0.5 * (u + sg * v)
            out[k + 1][at] = 0.5j * (u - sg * v)

    _legendre(lmax, spin, rings[0], dev, visit)
    for x in out:  # the m = 0 coefficients of real maps
        x[:lmax + 1] = x[:lmax + 1].real + 0j
    return out


def exact(case, seed):
    if case["kind"] == "batch":
        problems = _batch_problems(case)
        if sum(l for l, _ in problems) > 16000:
            return None
        maps, alm = [], []
        for (lmax, n), a in zip(problems, _batch_inputs(case, seed)):
            rings = _rings({"grid": "gauss", "nlat": lmax + 1, "nlon": 2 * lmax + 1})
            maps.append(_synthesis(lmax, 0, rings, a))
            alm.append(_analysis(lmax, 0, rings, maps[-1]))
        return {"maps": maps, "alm": alm}
    lmax, spin = case["lmax"], case["spin"]
    if lmax > 2100:
        return None
    rings, given = _rings(case), _inputs(case, seed)
    if case["kind"] == "pair":
        maps = _synthesis(lmax, spin, rings, given["alm"])
        return {"maps": maps, "alm": _analysis(lmax, spin, rings, maps)}
    if case["kind"] == "adjoint":
        alm = _analysis(lmax, spin, rings, given["maps"], weighted=False)
        return {"alm": alm, "maps": _synthesis(lmax, spin, rings, alm, weighted=True)}
    if case["kind"] == "jacobi":
        p = given["maps"][0]
        a = _analysis(lmax, 0, rings, [p])[0]
        for _ in range(3):
            r = p - _synthesis(lmax, 0, rings, [a])[0]
            a = a + _analysis(lmax, 0, rings, [r])[0]
        return {"alm": a, "residual": r}
    if case["kind"] == "deriv":  # Q + iU of E = sqrt(l (l + 1)) a, B = 0 at spin 1
        l, _ = _lm(lmax, given["alm"][0].device)
        e = [x for a in given["alm"] for x in (a * torch.sqrt(l * (l + 1.0)), torch.zeros_like(a))]
        return {"maps": _synthesis(lmax, 1, rings, e)}
    r = torch.stack(_synthesis(lmax, spin, rings, given["alm"])) - given["data"]
    g = torch.stack(_analysis(lmax, spin, rings, [2.0 * x for x in r], weighted=False))
    g[:, lmax + 1:] *= 2.0  # every m > 0 entry also stands for -m
    return {"loss": (r * r).sum(), "grad": g}
