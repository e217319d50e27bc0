"""The list walk's forms: several lanes per target over flat candidate lists,
and the targets whose candidates do not fit their segment, which keep chunk
records (a squeezed block of fluid: up to several times the usual number of
candidates).  Both against the FP64 oracle, element by element, with the
tolerances of test_gpu_list_eval (FP32 against FP64: 1e-4 of max|.|; pair
counts up to the pairs at the cut-off)."""
import numpy as np
import pytest

from paper_2104_00537_gb300 import cases, sph
from tests.test_gpu_list_eval import check_step_eval

pytestmark = pytest.mark.gpu


def squeezed(cell_mode, factor):
    """A small dam break whose fluid within 3 h of the column's centre is drawn
    towards it by the factor."""
    c = cases.dam_break(0.04, cell_mode=cell_mode)
    f = c.ptype == 0
    mid = 0.5 * (c.pos[f].min(0) + c.pos[f].max(0))
    d = c.pos - mid
    near = f & (np.linalg.norm(d, axis=1) < 3.0 * c.params["h"])
    c.pos[near] = mid + factor * d[near]
    return c


@pytest.mark.parametrize("cell_mode", [0, 1, 2])
@pytest.mark.parametrize("factor", [1.0, 0.8, 0.65])
@pytest.mark.parametrize("lanes,pair_once", [(0, 0), (1, 0), (4, 0), (0, 1)])
def test_flat_lists_and_kept_records(cell_mode, factor, lanes, pair_once):
    case = squeezed(cell_mode, factor)
    eng = sph.Engine.create(case)
    eng.set_options(pi_variant=5, pi_lanes=lanes, pair_once=pair_once, check_list=1)
    for stage in (0, 1):
        check_step_eval(case, eng, stage)
    eng.destroy()


@pytest.mark.parametrize("dp", [0.08, 0.013, 0.0105])
def test_targets_per_group(dp):
    """The smallest case (one target per lane group, a part of one block) and
    two sizes either side of where a group takes two targets."""
    case = cases.dam_break(dp)
    eng = sph.Engine.create(case)
    eng.set_options(use_graph=1)
    eng.step(2)
    check_step_eval(case, eng, 0, exact_pairs=False)
    eng.destroy()


@pytest.mark.parametrize("cell_mode", [0, 1, 2])
@pytest.mark.parametrize("slip", [0, 2])
def test_ghost_node_lists(cell_mode, slip):
    """mDBC boundary values from the ghost nodes' lists (variant 5) against the
    search of the cells' rows (variant 0), 20 steps of a moving tank.  Ghost
    offsets reach seven cells at cell_mode 2 (the lists' positions wrap at
    eight).  The sums are the same up to FP32 rounding (about 1e-6, times ten
    for the extrapolation to the wall); a missed neighbour shows at 1e-2."""
    c = cases.sloshing_tank(3000, 0.3, 0.03, 1.2, boundary_mode=1, mdbc_slip=slip,
                            cell_mode=cell_mode)
    out = []
    for variant in (5, 0):
        eng = sph.Engine.create(c)
        eng.set_options(pi_variant=variant)
        eng.step(20)
        out.append(eng.get_state())
        eng.destroy()
    a, b = out
    b_ = c.ptype != 0
    d = np.abs(a["rho"][b_] - b["rho"][b_]).max()
    assert d < 1e-3 * np.abs(b["rho"] - c.params["rho0"]).max(), d
    assert np.abs(a["vel"] - b["vel"]).max() < 1e-3 * np.abs(b["vel"]).max()
    assert np.abs(a["pos"] - b["pos"]).max() < 1e-3 * c.params["dp"]
