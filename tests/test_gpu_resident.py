"""The resident kernel (the form that runs of 16 or more steps of grids held in shared memory take)
against one launch per step: the same state, bit for bit.

Blocks of 64 columns exchange their borders through mailboxes and fold rows that several rounds of
warps share, so the shapes are those where this can go wrong: strips of 2, 63 and 64 columns, blocks
of 2 rows, of half a row per warp (at most 8 rows) and of one, two and several rounds, one block
that is its own neighbour, every side kind and its corners.  A run in place leaves the state in the
buffer it was in; an odd run of the other forms moves it to the other one.
"""
import numpy as np
import pytest

from paper_1909_04166_gb300 import lbm
from paper_1909_04166_gb300 import workloads as W

pytestmark = pytest.mark.gpu

RUNS = (17, 3, 16, 33)

# nx, ny, (left, right), (bottom, top): 0 periodic, 1 no-slip, 2 free-slip
SHAPES = [
    (2, 2, (0, 0), (0, 0)),
    (2, 9, (2, 1), (1, 2)),
    (64, 64, (0, 0), (0, 0)),
    (66, 5, (2, 2), (2, 2)),
    (63, 40, (1, 1), (0, 0)),
    (127, 3, (0, 0), (1, 2)),
    (128, 700, (1, 2), (2, 1)),
    (161, 481, (2, 2), (1, 1)),
    (257 + 63, 640, (0, 0), (0, 0)),
    (256, 1024, (0, 0), (1, 1)),
]


def run(case, precision, resident, runs=RUNS):
    """State and step counter after `runs`, and whether the runs of 16 and more stayed in place."""
    with lbm.Simulation(case, precision=precision) as sim:
        sim.init_case()
        if not resident:
            lbm.lbm_set_persistent(sim.ctx, 0)
        in_place = []
        for n in runs:
            before = lbm.lbm_state_device(sim.ctx)[0]
            sim.step(n)
            if n >= 16 and n % 2:
                in_place.append(lbm.lbm_state_device(sim.ctx)[0] == before)
        lbm.lbm_check(sim.ctx)
        raw, steps = sim.save_state()
    assert in_place and all(x == resident for x in in_place)
    return raw, steps


@pytest.mark.parametrize("precision", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("nx,ny,bx,by", SHAPES)
def test_resident_runs_match_single_steps(nx, ny, bx, by, precision):
    case = W.random_drop(nx, ny, seed=nx * 5 + ny, wall_x=bx[0], wall_x_hi=bx[1], wall_y=by[0],
                         wall_y_hi=by[1], rho_ratio=100.0, gravity=1e-6, marangoni=-2e-5)
    a, b = run(case, precision, True), run(case, precision, False)
    assert a[1] == b[1] == sum(RUNS)
    assert np.array_equal(a[0], b[0])


@pytest.mark.parametrize("ny", [66, 900])
@pytest.mark.parametrize("collision,sigma_model", [(1, 0), (0, 1), (1, 1)])
def test_resident_step_variants(collision, sigma_model, ny):
    case = W.random_drop(130, ny, seed=5, wall_y=1, rho_ratio=10.0, gravity=1e-6,
                         collision=collision, sigma_model=sigma_model, beta=0.4, psi0=0.2,
                         gradpsi_x=1e-3)
    assert np.array_equal(run(case, "fp32", True)[0], run(case, "fp32", False)[0])


@pytest.mark.parametrize("L0", [64, 200, 642])
def test_resident_imposed_flow_across_the_reversal(L0):
    case = W.shear_circle(L0=L0, u0=0.03)
    case.update(reverse_step=37)
    runs = (17, 60)               # the second run is split at the reversal
    out = []
    for resident in (True, False):
        raw, _ = run(case, "fp32", resident, runs)
        out.append(raw.view(np.float32).reshape(L0, -1, 18, 32)[:, :, 9:])
    assert np.array_equal(out[0], out[1])


def test_grids_beyond_shared_memory_and_one_node_strips_take_the_other_forms():
    for nx, ny in ((65, 40), (1, 30), (30, 1), (700, 900)):
        case = W.random_drop(nx, ny, seed=4, wall_y=1, rho_ratio=10.0)
        with lbm.Simulation(case, precision="fp32") as sim:
            sim.init_case()
            before = lbm.lbm_state_device(sim.ctx)[0]
            sim.step(17)
            assert lbm.lbm_state_device(sim.ctx)[0] != before
