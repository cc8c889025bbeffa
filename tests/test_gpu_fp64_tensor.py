"""The FP64 form with its contractions on the tensor cores (csrc/legendre_tc64.cu) against
the FP64 oracle, at the sizes where it takes over and where its tiles, blocks and
windows end, and over the exponent range of a double.

Tolerance: each Legendre value and each input enters with at most 2^-55 of its bound and
all sums of products are exact to 2^-56 of theirs, so the FP64 form's own bounds (1e-12
relative L2, 5e-12 of the largest value) hold unchanged.
"""
import numpy as np
import pytest

import oracle
from paper_1303_4945_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sht():
    from paper_1303_4945_gb300 import build

    build.build()
    from paper_1303_4945_gb300 import sht as m

    assert torch.cuda.is_available()
    return m


def both_ways(sht, geom, lmax, spin, alm, maps):
    plan = sht.sht_plan_create(geom, sht.sht_alm_create(lmax, lmax), spin, len(alm) // (2 if spin else 1), sht.SHT_FP64)
    a = [torch.from_numpy(x).cuda() for x in alm]
    p = [torch.full((geom.npix,), np.nan, dtype=torch.float64, device="cuda") for _ in alm]
    sht.sht_execute(plan, sht.SHT_SYNTHESIS, a, p)
    out = [torch.full((len(alm[0]),), complex(np.nan, np.nan), dtype=torch.complex128, device="cuda") for _ in alm]
    sht.sht_execute(plan, sht.SHT_ANALYSIS, out, [torch.from_numpy(x).cuda() for x in maps])
    assert plan.device_status() == 0
    return [x.cpu().numpy() for x in p], [x.cpu().numpy() for x in out]


def close(got, ref):
    for g, r in zip(got, ref):
        assert np.linalg.norm(g - r) <= 1e-12 * np.linalg.norm(r)
        assert np.max(np.abs(g - r)) <= 5e-12 * np.max(np.abs(r))


def rings_of(geom):
    r = geom.rings()
    return oracle.Rings(r["theta"], r["nphi"], r["phi0"], r["weight"], ofs=r["ofs"])


# (spin, ncomp, lmax, nlat): the lengths at which either direction takes over (one array
# 207 | 208 and 223 | 224, two 191 | 192, four 47 | 48), windows of 256 degrees full, one short
# and one over (lmax 255, 254, 256 at m = 0), tiles of 128 pairs (nlat 255 .. 258, 513)
@pytest.mark.parametrize("spin,ncomp,lmax,nlat", [
    (0, 1, 207, 210), (0, 1, 208, 255), (0, 1, 223, 224), (0, 1, 224, 256), (0, 1, 254, 258), (0, 1, 255, 257),
    (0, 1, 256, 513), (0, 2, 191, 193), (0, 2, 192, 258), (0, 2, 24, 26), (0, 3, 48, 257), (0, 4, 47, 50),
    (2, 1, 191, 258), (2, 1, 192, 255), (2, 1, 257, 300), (1, 2, 48, 49), (-3, 2, 60, 513), (5, 1, 24, 514)])
def test_edges_against_oracle(sht, spin, ncomp, lmax, nlat):
    rng = np.random.default_rng(1000 * lmax + nlat + spin)
    geom = sht.sht_geom_gauss(nlat, 2 * lmax + 1)
    rings = rings_of(geom)
    n = ncomp * (2 if spin else 1)
    alm = [inputs.gaussian_alm(rng, lmax, lmax, cl=inputs.cl_inverse_square, lmin=abs(spin)) for _ in range(n)]
    maps = [rng.standard_normal(geom.npix) for _ in range(n)]
    got_p, got_a = both_ways(sht, geom, lmax, spin, alm, maps)
    for k in range(0, n, 2 if spin else 1):
        sl = slice(k, k + (2 if spin else 1))
        close(got_p[sl], oracle.synthesis(spin, lmax, lmax, alm[sl], rings))
        close(got_a[sl], oracle.analysis(spin, lmax, lmax, maps[sl], rings))


# equal inputs of one sign (the longest runs of equal digits in the exact sums), values
# just below a power of two (the largest leading digit), and the ends of the exponent range
@pytest.mark.parametrize("value", [1.0, -1.0, 1.0 - 2.0**-53, 255.0 / 256, 3e250, 3e-250])
def test_equal_values_and_exponent_range(sht, value):
    lmax = 260
    geom = sht.sht_geom_gauss(262, 2 * lmax + 1)
    rings = rings_of(geom)
    _, m = inputs.lm_arrays(lmax, lmax)
    alm = np.where(m == 0, 1.0, 1.0 + 1.0j).astype(np.complex128)
    maps = np.ones(geom.npix)
    got_p, got_a = both_ways(sht, geom, lmax, 0, [value * alm], [value * maps])
    ref_a = oracle.analysis(0, lmax, lmax, [maps], rings)[0]
    close([got_p[0] / value], oracle.synthesis(0, lmax, lmax, [alm], rings))
    # only a_00 is not zero: the rest against the largest value
    assert np.max(np.abs(got_a[0] / value - ref_a)) <= 5e-12 * np.max(np.abs(ref_a))


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_inputs_stay_non_finite(sht, bad):
    lmax = 230
    geom = sht.sht_geom_gauss(300, 2 * lmax + 1)
    l, m = inputs.lm_arrays(lmax, lmax)
    alm = inputs.gaussian_alm(np.random.default_rng(5), lmax, lmax)
    alm[(l == 100) & (m == 7)] = bad
    maps = np.random.default_rng(6).standard_normal(geom.npix)
    maps[len(maps) // 2] = bad
    got_p, got_a = both_ways(sht, geom, lmax, 0, [alm], [maps])
    assert not np.isfinite(got_p[0]).any()  # the term reaches every pixel
    assert not np.isfinite(got_a[0][m < 20]).any()
