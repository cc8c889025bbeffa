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
