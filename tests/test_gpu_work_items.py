"""Work items whose size follows from the plan's: synthesis items of up to two tiles of
ring pairs (spin 0, one or two maps, tensor-core form) at ring counts around whole tiles,
with FP64 columns between them, and the limit of the call that allocates nothing, which
is one of the transform and not of the tiling that serves it."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MIX_L2 = 1e-10  # the mixed form's bound, relative L2 against the FP64 form


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


def rel(a, b):
    return float(torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(b))


@pytest.mark.parametrize("nlat", [256, 257, 511, 514, 770])
@pytest.mark.parametrize("ncomp", [1, 2])
def test_two_tile_items(sht, nlat, ncomp):
    lmax = 4800  # columns enough that one or two tiles each reach the rule's work per SM
    geom = sht.sht_geom_gauss(nlat, 96)
    lay = sht.sht_alm_create(lmax, lmax)
    mixed = sht.sht_plan_create(geom, lay, 0, ncomp, sht.SHT_MIXED)
    ref = sht.sht_plan_create(geom, lay, 0, ncomp, sht.SHT_FP64)
    alm = random_alm(lay, lmax, ncomp)
    maps = [torch.empty(geom.npix, dtype=torch.float64, device="cuda") for _ in range(ncomp)]
    want = [torch.empty_like(x) for x in maps]
    mixed.tensor_cores = True
    for flags in (0, sht.SHT_NO_POLAR_OPT):
        for x in maps:
            x.fill_(float("nan"))
        sht.sht_execute(mixed, sht.SHT_SYNTHESIS, alm, maps, flags)
        sht.sht_execute(ref, sht.SHT_SYNTHESIS, alm, want, flags)
        assert mixed.device_status() == 0
        for x, y in zip(maps, want):
            assert rel(x, y) <= MIX_L2
    mixed.tensor_cores = False  # the lists go back to single tiles
    sht.sht_execute(mixed, sht.SHT_SYNTHESIS, alm, maps, sht.SHT_NO_POLAR_OPT)
    for x, y in zip(maps, want):
        assert rel(x, y) <= MIX_L2


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


@pytest.mark.parametrize("nlat,lmax,ncomp", [(1, 0, 3), (2, 1, 4), (31, 33, 5), (254, 200, 16), (257, 260, 4), (511, 515, 8),
                                             (513, 518, 3), (1026, 600, 9), (700, 2100, 4)])
def test_analysis_of_more_than_two_maps(sht, nlat, lmax, ncomp):
    """Four maps at a time on the tensor cores: rings around whole tiles of 256 pairs,
    padded maps, FP64 columns (lmax >= 2000), no polar cut, added outputs."""
    geom = sht.sht_geom_gauss(nlat, 64)
    lay = sht.sht_alm_create(lmax, lmax)
    mixed = sht.sht_plan_create(geom, lay, 0, ncomp, sht.SHT_MIXED)
    ref = sht.sht_plan_create(geom, lay, 0, ncomp, sht.SHT_FP64)
    g = torch.Generator(device="cuda").manual_seed(4945)
    maps = [10.0 ** (2 * k) * torch.randn(geom.npix, dtype=torch.float64, device="cuda", generator=g) for k in range(-1, ncomp - 1)]
    got, want = ([torch.ones(lay.size(), dtype=torch.complex128, device="cuda") for _ in range(ncomp)] for _ in range(2))
    for flags in (0, sht.SHT_NO_POLAR_OPT, sht.SHT_ADD_OUTPUT):
        for type_ in (sht.SHT_ANALYSIS, sht.SHT_ADJOINT_SYNTHESIS):
            sht.sht_execute(mixed, type_, got, maps, flags)
            sht.sht_execute(ref, type_, want, maps, flags)
            assert mixed.device_status() == 0
            for x, y in zip(got, want):
                assert rel(x, y) <= MIX_L2


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("ncomp,tca", [(1, True), (2, True), (4, False), (8, False)])
def test_analysis_keeps_nan(sht, bad, ncomp, tca):
    """A pixel that is not finite, on the first ring (most columns' recursions never reach
    it) or the equator, leaves no finite coefficient of its map and every one of the others."""
    lmax = 299
    geom = sht.sht_geom_gauss(300, 601)
    lay = sht.sht_alm_create(lmax, lmax)
    plan = sht.sht_plan_create(geom, lay, 0, ncomp, sht.SHT_MIXED)
    plan.tensor_core_analysis = tca
    g = torch.Generator(device="cuda").manual_seed(7)
    for pos in (100, geom.npix // 2):
        maps = [torch.randn(geom.npix, dtype=torch.float64, device="cuda", generator=g) for _ in range(ncomp)]
        alm = [torch.zeros(lay.size(), dtype=torch.complex128, device="cuda") for _ in range(ncomp)]
        maps[0][pos] = bad
        sht.sht_execute(plan, sht.SHT_ANALYSIS, alm, maps)
        assert plan.device_status() == 0
        assert not torch.isfinite(torch.view_as_real(alm[0])[lmax + 1:]).any()
        assert not torch.isfinite(alm[0][: lmax + 1].real).any()
        assert all(torch.isfinite(torch.view_as_real(a)).all() for a in alm[1:])


@pytest.mark.parametrize("nlat,lmax", [(1, 0), (2, 1), (31, 33), (254, 47), (257, 64), (511, 300), (514, 65), (770, 515), (700, 2100)])
@pytest.mark.parametrize("ncomp", [1, 2])
def test_analysis_of_two_pairs_a_thread(sht, nlat, lmax, ncomp):
    """Rings around whole tiles of 256 pairs, last chunks of every length class, FP64
    columns (lmax >= 2000), no polar cut, added outputs."""
    geom = sht.sht_geom_gauss(nlat, 64)
    lay = sht.sht_alm_create(lmax, lmax)
    mixed = sht.sht_plan_create(geom, lay, 0, ncomp, sht.SHT_MIXED)
    mixed.set_tiling(2)
    ref = sht.sht_plan_create(geom, lay, 0, ncomp, sht.SHT_FP64)
    g = torch.Generator(device="cuda").manual_seed(512)
    maps = [torch.randn(geom.npix, dtype=torch.float64, device="cuda", generator=g) for _ in range(ncomp)]
    got, want = ([torch.ones(lay.size(), dtype=torch.complex128, device="cuda") for _ in range(ncomp)] for _ in range(2))
    for flags in (0, sht.SHT_NO_POLAR_OPT, sht.SHT_ADD_OUTPUT):
        for type_ in (sht.SHT_ANALYSIS, sht.SHT_ADJOINT_SYNTHESIS):
            sht.sht_execute(mixed, type_, got, maps, flags)
            sht.sht_execute(ref, type_, want, maps, flags)
            for x, y in zip(got, want):
                assert rel(x, y) <= MIX_L2


@pytest.mark.parametrize("nlat,lmax,ncomp", [(2, 2, 4), (31, 33, 3), (257, 260, 5), (513, 518, 4), (700, 2100, 3), (254, 100, 8)])
def test_spin_analysis_of_more_than_two_jobs(sht, nlat, lmax, ncomp):
    """Two E/B pairs at a time on the tensor cores, over tiles of 256 ring pairs."""
    geom = sht.sht_geom_gauss(nlat, 64)
    lay = sht.sht_alm_create(lmax, lmax)
    mixed = sht.sht_plan_create(geom, lay, 2, ncomp, sht.SHT_MIXED)
    ref = sht.sht_plan_create(geom, lay, 2, ncomp, sht.SHT_FP64)
    n = 2 * ncomp
    g = torch.Generator(device="cuda").manual_seed(37)
    maps = [torch.randn(geom.npix, dtype=torch.float64, device="cuda", generator=g) for _ in range(n)]
    got, want = ([torch.ones(lay.size(), dtype=torch.complex128, device="cuda") for _ in range(n)] for _ in range(2))
    for flags in (0, sht.SHT_NO_POLAR_OPT, sht.SHT_ADD_OUTPUT):
        for type_ in (sht.SHT_ANALYSIS, sht.SHT_ADJOINT_SYNTHESIS):
            sht.sht_execute(mixed, type_, got, maps, flags)
            sht.sht_execute(ref, type_, want, maps, flags)
            assert mixed.device_status() == 0
            for x, y in zip(got, want):
                assert rel(x, y) <= MIX_L2
