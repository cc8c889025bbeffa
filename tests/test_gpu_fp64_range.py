"""SHT_FP64 on inputs whose size varies over many powers of two inside one column: the
contraction in fixed point (csrc/legendre_tc64.cu) rounds relative to a column's largest
input, so what it cannot hold has to reach the IEEE kernels.  Results are compared term by
term, ring by ring or coefficient by coefficient, with the FP64 oracle.

Tolerance: 1e-11 of the terms that make up a result, the error of Lambda on these rings
and degrees in the plain recursion (1e-13 to 2e-12 in the IEEE kernels and the oracle);
fixed point alone loses 1e-7 and more here.
"""
import numpy as np
import pytest

import oracle
from paper_1303_4945_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LMAX, NLAT = 299, 300
TOL = 1e-11


@pytest.fixture(scope="module")
def sht():
    from paper_1303_4945_gb300 import build

    build.build()
    from paper_1303_4945_gb300 import sht as m

    assert torch.cuda.is_available()
    return m


def rings_of(geom):
    r = geom.rings()
    return oracle.Rings(r["theta"], r["nphi"], r["phi0"], r["weight"], ofs=r["ofs"])


def dev(x):
    return [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in x]


def execute(sht, plan, kind, how, alm, maps):
    """One transform by the plain call, the one that allocates nothing, a batch or a replayed graph."""
    if how == "batch":
        sht.sht_batch_execute(sht.sht_batch_create([plan]), kind, [alm], [maps])
    elif how == "noalloc":
        sht.sht_execute_noalloc(plan, kind, alm, maps)
    elif how == "graph":
        stream = torch.cuda.Stream()
        sht.sht_execute(plan, kind, alm, maps, 0, stream)
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            sht.sht_execute(plan, kind, alm, maps, 0, stream)
        for x in (maps if kind == sht.SHT_SYNTHESIS else alm):
            x.fill_(float("nan"))
        graph.replay()
    else:
        sht.sht_execute(plan, kind, alm, maps)
    torch.cuda.synchronize()


def amplitude(spin, m, theta):
    """|Lambda_lm| for l = m..LMAX, at its nodes the neighbouring degrees': its error is relative to that."""
    lam = np.maximum(np.abs(oracle.lambda_(spin, m, LMAX, theta)), np.abs(oracle.lambda_(-spin, m, LMAX, theta)))[m:]
    pad = np.pad(lam, 8)
    return np.max([pad[i:i + len(lam)] for i in range(17)], axis=0)


def steep(l, m):  # falls by 10^12 over 100 degrees
    return 10.0 ** (-0.12 * (l - m))


def band(l, m):  # nothing above l = 120, one degree below the last at m = 60
    return ((l <= 120) | ((m == 60) & (l == LMAX - 1))).astype(float)


def growing(l, m):  # no loss in fixed point, but every size
    return 10.0 ** (0.3 * (l - m))


@pytest.mark.parametrize("how", ["plain", "batch", "noalloc", "graph"])
@pytest.mark.parametrize("spin,ncomp,shape", [(0, 1, steep), (0, 1, band), (0, 3, steep), (0, 2, growing), (2, 1, steep), (2, 2, band), (-1, 1, steep)])
def test_synthesis_ring_by_ring(sht, spin, ncomp, shape, how):
    """One column of one m: each ring's values against the oracle's, over the sum of the
    sizes of that ring's terms (a value may cancel where Lambda has a node)."""
    geom = sht.sht_geom_gauss(NLAT, 2 * LMAX + 1)
    rings = rings_of(geom)
    plan = sht.sht_plan_create(geom, sht.sht_alm_create(LMAX, LMAX), spin, ncomp, sht.SHT_FP64)
    l, m = inputs.lm_arrays(LMAX, LMAX)
    rng = np.random.default_rng(99)
    n = ncomp * (2 if spin else 1)
    for col in (0, 60, 200):
        alm = []
        for _ in range(n):
            a = (rng.uniform(0.5, 1.0, len(l)) + 1j * rng.uniform(0.5, 1.0, len(l))) * shape(l, m) * (m == col) * (l >= abs(spin))
            alm.append(a.real.astype(complex) if col == 0 else a)
        got = [torch.full((geom.npix,), np.nan, dtype=torch.float64, device="cuda") for _ in alm]
        execute(sht, plan, sht.SHT_SYNTHESIS, how, dev(alm), got)
        assert plan.device_status() == 0
        per = 2 if spin else 1
        for k in range(0, n, per):
            ref = oracle.synthesis(spin, LMAX, LMAX, alm[k:k + per], rings)
            err = np.max([np.abs(g.cpu().numpy() - r).reshape(NLAT, -1).max(axis=1) for g, r in zip(got[k:k + per], ref)], axis=0)
            a = np.max([np.abs(x) for x in alm[k:k + per]], axis=0)[m == col]
            size = np.array([a @ amplitude(spin, col, t) for t in rings.theta])
            kept = size > 1e-60 * size.max()  # the polar cut drops rings below 2^-200
            assert (err[kept] <= TOL * size[kept]).all()


def bright_ring(geom, rng, spin):
    r = geom.rings()
    maps = []
    for _ in range(2 if spin else 1):
        x = rng.standard_normal(geom.npix)
        o = r["ofs"][20]  # theta = 0.21
        x[o:o + r["nphi"][20]] *= 1e10
        maps.append(x)
    return maps


@pytest.mark.parametrize("how", ["plain", "batch", "noalloc", "graph"])
@pytest.mark.parametrize("spin", [0, 2, 9, 37])
def test_analysis_beside_a_bright_ring(sht, spin, how):
    """The coefficients that a ring 10^10 times as bright as the rest does not reach."""
    geom = sht.sht_geom_gauss(NLAT, 2 * LMAX + 1)
    rings = rings_of(geom)
    plan = sht.sht_plan_create(geom, sht.sht_alm_create(LMAX, LMAX), spin, 1, sht.SHT_FP64)
    maps = bright_ring(geom, np.random.default_rng(5), spin)
    got = [torch.full((plan.alm.size(),), complex(np.nan, np.nan), dtype=torch.complex128, device="cuda") for _ in maps]
    execute(sht, plan, sht.SHT_ANALYSIS, how, got, dev(maps))
    assert plan.device_status() == 0
    ref = oracle.analysis(spin, LMAX, LMAX, maps, rings)
    l, m = inputs.lm_arrays(LMAX, LMAX)
    th = rings.theta[20]
    reach = np.concatenate([np.maximum(np.abs(oracle.lambda_(spin, k, LMAX, th)), np.abs(oracle.lambda_(-spin, k, LMAX, th)))[max(k, 0):]
                            for k in range(LMAX + 1)])
    free = (reach < 1e-30) & (l >= abs(spin))
    assert free.sum() > 5000
    for g, r in zip(got, ref):
        e = np.abs(g.cpu().numpy() - r)
        assert (e[free] <= TOL * np.sqrt(np.mean(np.abs(r[free]) ** 2))).all()
        assert np.linalg.norm(e) <= 1e-12 * np.linalg.norm(r)


@pytest.mark.parametrize("spin,ncomp", [(0, 1), (0, 2), (2, 1)])
def test_analysis_of_a_polar_cap(sht, spin, ncomp):
    """Rings of a cap only: at m = 150 the first degrees' Lambda is below 10^-30 on all of them."""
    full = sht.sht_geom_gauss(NLAT, 2 * LMAX + 1)
    geom = sht.sht_geom_subset(full, np.flatnonzero(full.rings()["theta"] < 0.6))
    rings = rings_of(geom)
    plan = sht.sht_plan_create(geom, sht.sht_alm_create(LMAX, LMAX), spin, ncomp, sht.SHT_FP64)
    rng = np.random.default_rng(8)
    n = ncomp * (2 if spin else 1)
    maps = [rng.standard_normal(geom.npix) for _ in range(n)]
    got = [torch.full((plan.alm.size(),), complex(np.nan, np.nan), dtype=torch.complex128, device="cuda") for _ in maps]
    sht.sht_execute(plan, sht.SHT_ANALYSIS, got, dev(maps))
    per = 2 if spin else 1
    l, m = inputs.lm_arrays(LMAX, LMAX)
    for k in range(0, n, per):
        ref = oracle.analysis(spin, LMAX, LMAX, maps[k:k + per], rings)
        for col in (60, 100, 150):
            s = (m == col) & (l >= abs(spin))
            size = np.max([np.abs(r[s]) for r in ref], axis=0)
            # neighbouring degrees' largest: a sum of random terms may cancel at one of them
            size = np.max([np.roll(size, i) for i in range(-4, 5)], axis=0)
            for g, r in zip(got[k:k + per], ref):
                e = np.abs(g.cpu().numpy()[s] - r[s])[4:-4]
                kept = size[4:-4] > 1e-80
                assert (e[kept] <= TOL * size[4:-4][kept]).all()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("ring", [0, 150])
def test_non_finite_values_as_in_ieee(sht, bad, ring):
    """A pixel or a coefficient that is not finite has the reach that it has in the IEEE
    kernels, and leaves the other arrays alone."""
    geom = sht.sht_geom_gauss(NLAT, 2 * LMAX + 1)
    lay = sht.sht_alm_create(LMAX, LMAX)
    plan = sht.sht_plan_create(geom, lay, 0, 2, sht.SHT_FP64)
    ieee = sht.sht_plan_create(geom, lay, 0, 2, sht.SHT_FP64)
    ieee.set_tiling(2)
    rng = np.random.default_rng(3)
    maps = [rng.standard_normal(geom.npix) for _ in range(2)]
    maps[0][ring * (2 * LMAX + 1) + 7] = bad
    out = []
    for p in (plan, ieee):
        a = [torch.zeros(lay.size(), dtype=torch.complex128, device="cuda") for _ in range(2)]
        sht.sht_execute(p, sht.SHT_ANALYSIS, a, dev(maps))
        out.append([x.cpu().numpy() for x in a])
    assert not np.isfinite(out[0][0]).all() and np.isfinite(out[0][1]).all()
    for x, y in zip(*out):
        f = np.isfinite(y)
        # (the IEEE tiling of the reference is coarser: its first terms start with its tiles)
        assert (np.isfinite(x) >= f).all()
        assert np.max(np.abs(x[f] - y[f]), initial=0.0) <= 1e-12 * max(1e-300, np.max(np.abs(y[f]), initial=0.0))
