"""The analysis settings of a plan (tiling, tensor-core analysis, autotuning): what a call
sets is what runs, and a plan returns to a setting in the state it had there.  A plan's
workspace counts its work lists and partial sums, so it shows which lists it holds.
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


def make(sht, lmax, nlat, spin, ncomp, precision):
    return sht.sht_plan_create(sht.sht_geom_gauss(nlat, 2 * lmax + 2), sht.sht_alm_create(lmax, lmax), spin, ncomp, precision)


@pytest.mark.parametrize("precision", [0, 1])
def test_workspace_follows_the_lists(sht, precision):
    """Changing a setting there and back leaves the workspace as it was."""
    plan = make(sht, 200, 600, 0, 1, precision)
    plan.set_tiling(8)
    eight = plan.workspace()
    plan.set_tiling(4)
    plan.set_tiling(8)
    assert plan.workspace() == eight
    if precision:
        plan.fp64_columns = 9
        nine = plan.workspace()
        plan.fp64_columns = 3
        plan.fp64_columns = 9
        assert plan.workspace() == nine
@pytest.mark.parametrize("spin,ncomp", [(2, 1), (2, 2)])
def test_lists_follow_the_kernel(sht, spin, ncomp):
    """292 rings are two tiles of 128 pairs: one item of the tensor-core analysis, two of
    the double-float one."""
    partials = {}
    for how in ("tiling", "switch", "autotune"):
        plan = make(sht, 144, 292, spin, ncomp, sht.SHT_MIXED)
        base = plan.workspace()
        if how == "tiling":
            plan.set_tiling(2)
            plan.set_tiling(1)
        elif how == "switch":
            plan.tensor_core_analysis = True
            plan.tensor_core_analysis = False
        else:
            plan.autotune(torch.cuda.current_stream())
            if plan.tensor_core_analysis:
                plan.tensor_core_analysis = False
            plan.set_tiling(1)
        assert plan.tiling()[0] == 1 and not plan.tensor_core_analysis
        partials[how] = plan.workspace() - base
    assert partials["switch"] == partials["tiling"] == partials["autotune"]


def test_fp64_tilings_come_back(sht):
    """The tensor-core contraction of an FP64 plan (tiles of 128 pairs) is the default
    tiling's, whichever way a caller returns to it."""
    plan = make(sht, 511, 1100, 0, 2, sht.SHT_FP64)
    cur, cands = plan.tiling()
    own = plan.workspace()
    plan.set_tiling(cur)
    assert plan.workspace() == own
    plan.set_tiling(cands[1])
    ieee = plan.workspace()
    assert ieee != own
    plan.set_tiling(cur)
    assert plan.workspace() == own
    plan.set_tiling(cands[1])
    plan.autotune(torch.cuda.current_stream())
    assert plan.workspace() == own  # three times as fast here (lmax 767: 3826 against 1228 us)
    batch = sht.sht_batch_create([plan])
    plan.set_tiling(plan.tiling()[0])
    assert plan.workspace() == own
    other = [c for c in cands if c != plan.tiling()[0]][0]
    with pytest.raises(sht.ShtError):
        plan.set_tiling(other)
    assert plan.workspace() == own
    del batch
    plan.set_tiling(other)


def test_a_refused_tiling_changes_nothing(sht):
    """A value that the tensor-core analysis refuses leaves the limit of the call that
    allocates nothing as it was: the former default tiling's until one is chosen."""
    lmax = 1350
    plan = make(sht, lmax, lmax + 1, 0, 1, sht.SHT_MIXED)
    plan.tensor_core_analysis = True
    with pytest.raises(sht.ShtError):
        plan.set_tiling(4)
    plan.tensor_core_analysis = False
    plan.fp64_columns = 0  # builds the lists again
    m = [torch.zeros(plan.geom.npix, dtype=torch.float64, device="cuda")]
    a = [torch.zeros(plan.alm.size(), dtype=torch.complex128, device="cuda")]
    sht.sht_execute_noalloc(plan, sht.SHT_ANALYSIS, a, m)


def analysis(sht, plan, maps):
    out = [torch.full((plan.alm.size(),), complex(float("nan")), dtype=torch.complex128, device="cuda") for _ in maps]
    sht.sht_execute(plan, sht.SHT_ANALYSIS, out, maps)
    assert plan.device_status() == 0
    return out


def close(x, y, tol):
    return float(torch.linalg.vector_norm(x - y)) <= tol * float(torch.linalg.vector_norm(y))


# three or more jobs: one and several tiles of 256 pairs, padded jobs, several groups
@pytest.mark.parametrize("spin,ncomp,nlat", [(0, 3, 31), (0, 16, 300), (2, 3, 520), (-1, 8, 300)])
def test_double_float_on_request(sht, spin, ncomp, nlat):
    """Plans of more than two jobs contract their analysis on the tensor cores and say so;
    0 takes every item to double-float."""
    geom, lay = sht.sht_geom_gauss(nlat, 64), sht.sht_alm_create(299, 299)
    plan, ref = (sht.sht_plan_create(geom, lay, spin, ncomp, sht.SHT_MIXED) for _ in range(2))
    g = torch.Generator(device="cuda").manual_seed(nlat)
    maps = [torch.randn(geom.npix, dtype=torch.float64, device="cuda", generator=g) for _ in range(plan.narrays)]
    assert plan.tensor_core_analysis
    a = analysis(sht, plan, maps)
    plan.tensor_core_analysis = False
    assert not plan.tensor_core_analysis and ref.tensor_core_analysis
    b = analysis(sht, plan, maps)
    assert any(not torch.equal(x, y) for x, y in zip(a, b))
    assert all(close(x, y, 1e-10) for x, y in zip(a, b))
    with pytest.raises(sht.ShtError):
        plan.tensor_core_analysis = True


@pytest.mark.parametrize("spin,ncomp", [(0, 1), (0, 2), (2, 1)])
def test_ieee_on_request(sht, spin, ncomp):
    """An FP64 plan says which contraction it has; 0 keeps the IEEE one, for both directions."""
    plan = make(sht, 300, 302, spin, ncomp, sht.SHT_FP64)
    small = make(sht, 20, 22, spin, ncomp, sht.SHT_FP64)
    assert plan.tensor_cores and plan.tensor_core_analysis
    assert not small.tensor_cores and not small.tensor_core_analysis
    g = torch.Generator(device="cuda").manual_seed(spin)
    alm = [torch.randn(plan.alm.size(), dtype=torch.complex128, device="cuda", generator=g) for _ in range(plan.narrays)]
    maps = [[torch.empty(plan.geom.npix, dtype=torch.float64, device="cuda") for _ in alm] for _ in range(2)]
    sht.sht_execute(plan, sht.SHT_SYNTHESIS, alm, maps[0])
    a = analysis(sht, plan, maps[0])
    plan.tensor_cores = False
    plan.tensor_core_analysis = False
    assert not plan.tensor_cores and not plan.tensor_core_analysis
    sht.sht_execute(plan, sht.SHT_SYNTHESIS, alm, maps[1])
    b = analysis(sht, plan, maps[0])
    for x, y in zip(maps[0] + a, maps[1] + b):
        assert not torch.equal(x, y) and close(x, y, 1e-12)
    plan.set_tiling(plan.tiling()[1][1])  # (for good: no tiling and no timing returns to the tensor cores)
    plan.set_tiling(plan.tiling()[1][0])
    plan.autotune(torch.cuda.current_stream())
    assert not plan.tensor_core_analysis
    for on in ("tensor_cores", "tensor_core_analysis"):
        with pytest.raises(sht.ShtError) as e:
            setattr(plan, on, True)
        assert e.value.code == sht.SHT_ERR_INVALID_ARG


def test_fp64_synthesis_of_few_columns_or_rings(sht):
    """One array's synthesis goes to the tensor cores where its columns' warps of ring pairs
    reach one per SM quarter; results are the IEEE sums' either way."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for lmax, nlat, mmax, on in ((255, 256, 255, 1024 >= 4 * sms), (255, 40, 255, 256 >= 4 * sms), (1023, 300, 40, 205 >= 4 * sms), (1023, 300, 1023, 5120 >= 4 * sms)):
        geom = sht.sht_geom_gauss(nlat, 2 * mmax + 2)
        plan = sht.sht_plan_create(geom, sht.sht_alm_create(lmax, mmax), 0, 1, sht.SHT_FP64)
        assert plan.tensor_cores == on
        g = torch.Generator(device="cuda").manual_seed(nlat)
        alm = [torch.randn(plan.alm.size(), dtype=torch.complex128, device="cuda", generator=g)]
        maps = [torch.empty(geom.npix, dtype=torch.float64, device="cuda") for _ in range(2)]
        sht.sht_execute(plan, sht.SHT_SYNTHESIS, alm, maps[:1])
        plan.tensor_cores = False
        sht.sht_execute(plan, sht.SHT_SYNTHESIS, alm, maps[1:])
        assert close(maps[0], maps[1], 1e-12)
