"""The double-float synthesis of many maps, whose kernels keep the recursion's difference
form for rings next to a pole in every warp, in none or in a second copy of their loops,
by the plan's rings and lmax (mix_polar_form): each against the FP64 form, and a batch of
them against the plans' own calls.  Tolerance: the mixed form's 1e-10.
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


def random_alm(lay, n, spin):
    g = torch.Generator(device="cuda").manual_seed(spin + n)
    return [torch.randn(lay.size(), dtype=torch.complex128, device="cuda", generator=g) for _ in range(n)]


@pytest.mark.parametrize("spin,ncomp", [(0, 9), (0, 16), (2, 5), (-1, 8)])
def test_forms(sht, spin, ncomp):
    plans, alms, maps = [], [], []
    # rings at the poles; none within 0.005 rad; some, lmax beyond the line between the two
    for geom, lay in ((sht.sht_geom_ecp(sht.SHT_ECP_CC, 131, 96), sht.sht_alm_create(64, 40)),
                      (sht.sht_geom_gauss(101, 96), sht.sht_alm_create(99, 40)),
                      (sht.sht_geom_gauss(1300, 32), sht.sht_alm_create(1250, 12))):
        plan = sht.sht_plan_create(geom, lay, spin, ncomp, sht.SHT_MIXED)
        ref = sht.sht_plan_create(geom, lay, spin, ncomp, sht.SHT_FP64)
        alm = random_alm(lay, plan.narrays, abs(spin))
        got, want = ([torch.full((geom.npix,), float("nan"), dtype=torch.float64, device="cuda") for _ in alm] for _ in range(2))
        sht.sht_execute(plan, sht.SHT_SYNTHESIS, alm, got)
        sht.sht_execute(ref, sht.SHT_SYNTHESIS, alm, want)
        for g, w in zip(got, want):
            assert torch.linalg.vector_norm(g - w) <= 1e-10 * torch.linalg.vector_norm(w)
        plans.append(plan)
        alms.append(alm)
        maps.append(got)
    out = [[torch.empty_like(x) for x in m] for m in maps]
    sht.sht_batch_execute(sht.sht_batch_create(plans), sht.SHT_SYNTHESIS, alms, out)
    for a, b in zip(out, maps):
        assert all(torch.equal(x, y) for x, y in zip(a, b))
