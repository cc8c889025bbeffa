"""Ring FFTs of calls with few rings, which give a ring more threads than calls of many (and
batches) do: the same results bit for bit, over ring lengths of every engine (mixed
radix, Rader, Bluestein).
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sht():
    from paper_1303_4945_gb300 import build

    build.build()
    from paper_1303_4945_gb300 import sht as m

    assert torch.cuda.is_available()
    return m


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nlon", [96, 128, 129, 512, 600, 613, 1000, 1024, 1025, 2048, 2055, 4095, 8191])
def test_own_call_and_batch_agree(sht, nlon, precision):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for nlat in (20, 3 * sms):  # below one ring pair per SM, between one and two
        geom = sht.sht_geom_gauss(nlat, nlon)
        lay = sht.sht_alm_create(19, 19)
        plan = sht.sht_plan_create(geom, lay, 0, 1, precision)
        g = torch.Generator(device="cuda").manual_seed(nlon)
        alm = [torch.randn(lay.size(), dtype=torch.complex128, device="cuda", generator=g)]
        maps = [torch.randn(geom.npix, dtype=torch.float64, device="cuda", generator=g)]
        batch = sht.sht_batch_create([plan])
        m = [torch.empty_like(maps[0]) for _ in range(2)]
        a = [torch.empty_like(alm[0]) for _ in range(2)]
        sht.sht_execute(plan, sht.SHT_SYNTHESIS, alm, [m[0]])
        sht.sht_batch_execute(batch, sht.SHT_SYNTHESIS, [alm], [[m[1]]])
        sht.sht_execute(plan, sht.SHT_ANALYSIS, [a[0]], maps)
        sht.sht_batch_execute(batch, sht.SHT_ANALYSIS, [[a[1]]], [maps])
        assert torch.equal(m[0], m[1]) and torch.equal(torch.view_as_real(a[0]), torch.view_as_real(a[1]))
