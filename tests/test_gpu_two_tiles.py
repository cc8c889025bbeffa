"""Synthesis items of two tiles (one or two spin-0 maps, tensor-core form): plans whose 128-pair
tiles reach the rule's 40 per SM on this GPU, whatever its SM count, against the FP64 form
and, on three rings, the FP64 oracle.  Tolerance: the mixed form's 1e-10.
"""
import numpy as np
import pytest

import oracle
from paper_1303_4945_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.fixture(scope="module")
def sht():
    from paper_1303_4945_gb300 import build

    build.build()
    from paper_1303_4945_gb300 import sht as m

    assert torch.cuda.is_available()
    return m


@pytest.mark.parametrize("nlat", [256, 257, 514])  # one tile per m; a second of one pair; three
@pytest.mark.parametrize("ncomp", [1, 2])
def test_two_tiles(sht, nlat, ncomp):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    lmax = 44 * sms
    geom = sht.sht_geom_gauss(nlat, 64)
    npairs = geom.info()[2]
    first = np.asarray(sht.sht_geom_polar_cut(geom, lmax, 0, np.arange(lmax + 1))[0])
    assert np.sum((npairs + 127) // 128 - first // 128) >= 40 * sms
    lay = sht.sht_alm_create(lmax, lmax)
    mixed = sht.sht_plan_create(geom, lay, 0, ncomp, sht.SHT_MIXED)
    mixed.tensor_cores = True
    ref = sht.sht_plan_create(geom, lay, 0, ncomp, sht.SHT_FP64)
    ref.tensor_cores = False  # IEEE sums
    rng = np.random.default_rng(nlat)
    alm = [inputs.gaussian_alm(rng, lmax, lmax) for _ in range(ncomp)]
    src = [torch.from_numpy(a).cuda() for a in alm]
    got, want = ([torch.full((geom.npix,), np.nan, dtype=torch.float64, device="cuda") for _ in alm] for _ in range(2))
    for flags in (0, sht.SHT_NO_POLAR_OPT):
        sht.sht_execute(mixed, sht.SHT_SYNTHESIS, src, got, flags)
        sht.sht_execute(ref, sht.SHT_SYNTHESIS, src, want, flags)
        assert mixed.device_status() == 0
        for g, w in zip(got, want):
            assert torch.linalg.vector_norm(g - w) <= TOL * torch.linalg.vector_norm(w)
    r = geom.rings()
    rings = oracle.Rings(r["theta"], r["nphi"], r["phi0"], r["weight"], ofs=r["ofs"])
    for y in (0, nlat // 3, nlat // 2):
        px = slice(r["ofs"][y], r["ofs"][y] + 64)
        o = oracle.synthesis(0, lmax, lmax, alm[-1], rings, rings_sel=[y])[0][px]
        assert np.max(np.abs(got[-1].cpu().numpy()[px] - o)) <= TOL * np.max(np.abs(o))
