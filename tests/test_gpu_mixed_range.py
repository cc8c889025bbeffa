"""The mixed form's analysis of more than two maps or E/B pairs on rings whose values vary
over many powers of two: the digit contraction (csrc/legendre_tc_ana.cu) rounds relative to
the brightest ring, so items it cannot hold run in double-float.  Coefficients are compared
one by one with the FP64 oracle.

Tolerance: the mixed form's 1e-10, of the coefficients themselves; the digits alone lose
1e-5 and more here.
"""
import numpy as np
import pytest

import oracle
from paper_1303_4945_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LMAX, NLAT = 299, 300
TOL = 1e-10


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


def analysis(sht, geom, spin, ncomp, maps, how="plain"):
    plan = sht.sht_plan_create(geom, sht.sht_alm_create(LMAX, LMAX), spin, ncomp, sht.SHT_MIXED)
    src = [torch.from_numpy(x).cuda() for x in maps]
    out = [torch.full((plan.alm.size(),), complex(np.nan, np.nan), dtype=torch.complex128, device="cuda") for _ in maps]
    if how == "batch":
        sht.sht_batch_execute(sht.sht_batch_create([plan]), sht.SHT_ANALYSIS, [out], [src])
    elif how == "noalloc":
        sht.sht_execute_noalloc(plan, sht.SHT_ANALYSIS, out, src)
    else:
        sht.sht_execute(plan, sht.SHT_ANALYSIS, out, src)
    torch.cuda.synchronize()
    assert plan.device_status() == 0
    return [x.cpu().numpy() for x in out]


def lam(spin, m, theta):
    return np.maximum(np.abs(oracle.lambda_(spin, m, LMAX, theta)), np.abs(oracle.lambda_(-spin, m, LMAX, theta)))[m:]


@pytest.mark.parametrize("how", ["plain", "batch", "noalloc"])
@pytest.mark.parametrize("spin,ncomp", [(0, 3), (0, 5), (2, 3)])
def test_beside_a_bright_ring(sht, spin, ncomp, how):
    geom = sht.sht_geom_gauss(NLAT, 2 * LMAX + 1)
    rings = rings_of(geom)
    rng = np.random.default_rng(5)
    n = ncomp * (2 if spin else 1)
    maps = [rng.standard_normal(geom.npix) for _ in range(n)]
    bright = 2 if spin else 1
    for x in maps[-bright:]:  # of the last job only
        x[20 * (2 * LMAX + 1):21 * (2 * LMAX + 1)] *= 1e10
    got = analysis(sht, geom, spin, ncomp, maps, how)
    l, m = inputs.lm_arrays(LMAX, LMAX)
    reach = np.concatenate([lam(spin, k, rings.theta[20]) for k in range(LMAX + 1)])
    free = (reach < 1e-30) & (l >= abs(spin))
    assert free.sum() > 5000
    for k in (0, n - bright):
        ref = oracle.analysis(spin, LMAX, LMAX, maps[k:k + bright], rings)
        for g, r in zip(got[k:k + bright], ref):
            e = np.abs(g - r)
            assert (e[free] <= TOL * np.sqrt(np.mean(np.abs(r[free]) ** 2))).all()
            assert np.linalg.norm(e) <= TOL * np.linalg.norm(r)


@pytest.mark.parametrize("spin,ncomp", [(0, 4), (2, 4)])
def test_of_a_polar_cap(sht, spin, ncomp):
    """Rings of a cap only: at m = 60 the first degrees' Lambda is below 10^-12 on all of them."""
    full = sht.sht_geom_gauss(NLAT, 2 * LMAX + 1)
    geom = sht.sht_geom_subset(full, np.flatnonzero(full.rings()["theta"] < 0.6))
    rings = rings_of(geom)
    rng = np.random.default_rng(8)
    n = ncomp * (2 if spin else 1)
    maps = [rng.standard_normal(geom.npix) for _ in range(n)]
    got = analysis(sht, geom, spin, ncomp, maps)
    per = 2 if spin else 1
    l, m = inputs.lm_arrays(LMAX, LMAX)
    ref = oracle.analysis(spin, LMAX, LMAX, maps[:per], rings)
    for col in (30, 60):
        s = (m == col) & (l >= abs(spin))
        size = np.max([np.abs(r[s]) for r in ref], axis=0)
        size = np.max([np.roll(size, i) for i in range(-4, 5)], axis=0)
        for g, r in zip(got[:per], ref):
            assert (np.abs(g[s] - r[s])[4:-4] <= TOL * size[4:-4]).all()
