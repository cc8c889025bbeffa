"""Rings without a mirror image on the other side of the equator, next to both poles, at
sizes where the recursion's per-pair tables (bounds, join records, difference form) decide
the result: both directions against the FP64 oracle, ring by ring.

Tolerances, of a ring's largest value: 1e-10, the per-ring bound that the mixed form is
built to; the oracle's own plain recursion keeps 2e-11 at theta = 3e-4, lmax 4095.
"""
import numpy as np
import pytest

import oracle
from paper_1303_4945_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MMAX, NPHI = 40, 97


@pytest.fixture(scope="module")
def sht():
    from paper_1303_4945_gb300 import build

    build.build()
    from paper_1303_4945_gb300 import sht as m

    assert torch.cuda.is_available()
    return m


def run(sht, theta, lmax, spin, ncomp, precision):
    """Synthesis per ring (map rows) and analysis, with the oracle's results."""
    n = len(theta)
    ofs = np.arange(n, dtype=np.int64) * NPHI
    nphi, phi0, weight = np.full(n, NPHI, np.int32), 0.1 * np.arange(n), np.linspace(0.5, 1.5, n)
    geom = sht.sht_geom_general(theta, nphi, phi0, ofs, None, weight)
    assert geom.info()[2] == n  # no two of the rings are mirror images
    rings = oracle.Rings(theta, nphi, phi0, weight, ofs=ofs)
    plan = sht.sht_plan_create(geom, sht.sht_alm_create(lmax, MMAX), spin, ncomp, precision)
    rng = np.random.default_rng(lmax + spin)
    narr = ncomp * (2 if spin else 1)
    alm = [inputs.gaussian_alm(rng, lmax, MMAX, lmin=abs(spin)) for _ in range(narr)]
    maps = [rng.standard_normal(n * NPHI) for _ in range(narr)]
    got_p = [torch.full((n * NPHI,), np.nan, dtype=torch.float64, device="cuda") for _ in alm]
    got_a = [torch.full((len(alm[0]),), complex(np.nan, np.nan), dtype=torch.complex128, device="cuda") for _ in alm]
    sht.sht_execute(plan, sht.SHT_SYNTHESIS, [torch.from_numpy(x).cuda() for x in alm], got_p)
    sht.sht_execute(plan, sht.SHT_ANALYSIS, got_a, [torch.from_numpy(x).cuda() for x in maps])
    assert plan.device_status() == 0
    per = 2 if spin else 1
    ref_p, ref_a = [], []
    for k in range(0, narr, per):
        ref_p += oracle.synthesis(spin, lmax, MMAX, alm[k:k + per], rings)
        ref_a += oracle.analysis(spin, lmax, MMAX, maps[k:k + per], rings)
    rows = [(g.cpu().numpy().reshape(n, NPHI), r.reshape(n, NPHI)) for g, r in zip(got_p, ref_p)]
    return rows, [(g.cpu().numpy(), r) for g, r in zip(got_a, ref_a)]


def ring_errors(rows):
    """Largest error of each ring over its largest value (of the pair of maps at spin s)."""
    err = np.max([np.abs(g - r).max(axis=1) for g, r in rows], axis=0)
    return err / np.max([np.abs(r).max(axis=1) for _, r in rows], axis=0)


def rings_near_both_poles(lo, hi, n):
    south = np.pi - np.linspace(lo, hi, n)
    return np.sort(np.concatenate([np.linspace(lo, hi, 9)[1:-1] * 1.003, [0.7, 1.3], south]))


@pytest.mark.parametrize("spin,ncomp", [(0, 1), (0, 2), (2, 1), (-1, 2)])
@pytest.mark.parametrize("lmax", [3000, 4095])
def test_fp64_form(sht, lmax, spin, ncomp):
    rows, alm = run(sht, rings_near_both_poles(3e-4, 6e-4, 60), lmax, spin, ncomp, sht.SHT_FP64)
    assert ring_errors(rows).max() <= 1e-10
    for g, r in alm:
        assert np.max(np.abs(g - r)) <= 1e-10 * np.max(np.abs(r))


@pytest.mark.parametrize("spin,ncomp", [(0, 1), (0, 2), (0, 4), (1, 1), (2, 1), (2, 3)])
def test_mixed_form(sht, spin, ncomp):
    rows, alm = run(sht, rings_near_both_poles(1.5e-3, 6.5e-3, 60), 1535, spin, ncomp, sht.SHT_MIXED)
    assert ring_errors(rows).max() <= 1e-10
    for g, r in alm:
        assert np.max(np.abs(g - r)) <= 1e-10 * np.max(np.abs(r))


def test_south_pole_alone(sht):
    """A ring at theta = pi without one at 0: only the column that survives there."""
    for spin in (0, 1, 2):
        rows, _ = run(sht, np.array([0.4, 1.2, np.pi]), 60, spin, 1, sht.SHT_FP64)
        assert ring_errors(rows).max() <= 1e-12
