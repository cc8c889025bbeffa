"""The limit of the call that allocates nothing is one of the transform, not of the
tiling that serves it."""
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


def random_alm(lay, lmax, n):
    g = torch.Generator(device="cuda").manual_seed(1303)
    out = []
    for _ in range(n):
        a = torch.randn(lay.size(), dtype=torch.complex128, device="cuda", generator=g)
        a[: lmax + 1].imag.zero_()  # m = 0
        out.append(a)
    return out


@pytest.mark.parametrize("precision", [0, 1])
def test_noalloc_limit_is_the_transforms(sht, precision):
    lmax = 1350  # phases and the sums of 512-pair tiles take 55.7 MiB, of 256-pair tiles 69.7
    geom = sht.sht_geom_gauss(lmax + 1, 2 * lmax + 2)
    lay = sht.sht_alm_create(lmax, lmax)
    plan = sht.sht_plan_create(geom, lay, 0, 1, precision)
    alm = random_alm(lay, lmax, 1)
    m = [torch.empty(geom.npix, dtype=torch.float64, device="cuda")]
    sht.sht_execute(plan, sht.SHT_SYNTHESIS, alm, m)
    want, got = [torch.empty_like(alm[0])], [torch.empty_like(alm[0])]
    sht.sht_execute(plan, sht.SHT_ANALYSIS, want, m)
    sht.sht_execute_noalloc(plan, sht.SHT_ANALYSIS, got, m)
    assert torch.equal(torch.view_as_real(want[0]), torch.view_as_real(got[0]))
    plan.set_tiling(2)  # a tiling asked for counts with its own sums
    code = 0
    try:  # (an exception kept here would keep the plan's memory past the test)
        sht.sht_execute_noalloc(plan, sht.SHT_ANALYSIS, got, m)
    except sht.ShtError as e:
        code = e.code
    assert code == sht.SHT_ERR_UNSUPPORTED
