"""The resident kernel (the form that runs of 16 or more steps of grids held in shared memory take)
against one launch per step: the same state, bit for bit.

Blocks of 64 columns exchange their borders through mailboxes and fold rows that several rounds of
warps share, so the shapes are those where this can go wrong: strips of 1, 2, 63 and 64 columns, blocks
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
    (65, 40, (0, 0), (0, 0)),           # a last strip of one column
    (129, 200, (0, 0), (2, 1)),
    (65, 33, (1, 2), (0, 0)),
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


# grids of blocks that take two rounds of 16 rows (27, 17 = 16 + 1, 22 rows), beside no-slip and
# free-slip sides: the first row of the second round is pushed into from both
@pytest.mark.parametrize("precision", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("nx,ny,bx,by", [
    (512, 512, (1, 1), (0, 0)),
    (256, 640, (1, 1), (1, 1)),
    (256, 640, (1, 2), (2, 1)),
    (256, 640, (2, 1), (1, 2)),
    (320, 640, (2, 2), (1, 1)),
])
def test_rounds_beside_side_walls(nx, ny, bx, by, precision):
    test_resident_runs_match_single_steps(nx, ny, bx, by, precision)


@pytest.mark.parametrize("bx", [(1, 1), (1, 2)])
def test_three_rounds_beside_side_walls(bx):
    """Blocks of 35 rows; and with the interface lattice alone of 43 rows."""
    test_resident_runs_match_single_steps(128, 2600, bx, (1, 1), "fp32")
    case = W.shear_circle(L0=640, u0=0.03)
    case.update(wall_x=bx[0], wall_x_hi=bx[1])
    out = [run(case, "fp32", r, (17, 33))[0].view(np.float32).reshape(640, -1, 18, 32)[:, :, 9:]
           for r in (True, False)]
    assert np.array_equal(out[0], out[1])


def test_rounds_of_a_batch_beside_side_walls():
    cases = [W.random_drop(nx, ny, seed=nx, wall_x=bx, wall_x_hi=hi, wall_y=1, rho_ratio=50.0,
                           gravity=1e-6)
             for nx, ny, bx, hi in ((200, 220, 1, 1), (90, 250, 1, 2), (130, 180, 2, 1))] * 12
    for precision in ("fp32", "fp16"):
        outs = []
        for resident in (True, False):
            with lbm.Batch(cases, precision=precision, layout=lbm.LBM_BATCH_AS_GIVEN) as b:
                b.init_all()
                if not resident:
                    lbm.lbm_batch_set_persistent(b.b, 0)
                b.step(65)
                outs.append([b.populations(i) for i in range(len(cases))])
        for (ga, fa), (gb, fb) in zip(*outs):
            assert np.array_equal(ga, gb) and np.array_equal(fa, fb)


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


@pytest.mark.parametrize("layout", [lbm.LBM_BATCH_AS_GIVEN, lbm.LBM_BATCH_FEWEST_COLUMNS])
@pytest.mark.parametrize("precision", ["fp32", "fp16", "bf16"])
def test_resident_batches_match_graph_replays(precision, layout):
    """Cases of several waves, among them single-column strips and a case of one block."""
    cases = W.ensemble(40) + [
        W.random_drop(nx, ny, seed=nx, wall_x=bx, wall_y=by, rho_ratio=50.0, gravity=1e-6)
        for nx, ny, bx, by in ((65, 70, 0, 0), (193, 65, 0, 2), (129, 65, 2, 1), (2, 2, 0, 0),
                               (64, 300, 1, 0), (33, 20, 0, 1))]
    outs = []
    for resident in (True, False):
        with lbm.Batch(cases, precision=precision, layout=layout) as b:
            b.init_all()
            if not resident:
                lbm.lbm_batch_set_persistent(b.b, 0)
            for n in (65, 1, 2, 80):
                b.step(n)
            lbm.lbm_batch_check(b.b)
            outs.append([b.populations(i) for i in range(len(cases))])
    for (ga, fa), (gb, fb) in zip(*outs):
        assert np.array_equal(ga, gb) and np.array_equal(fa, fb)


@pytest.mark.parametrize("collision,sigma_model", [(1, 0), (0, 1), (1, 1)])
def test_resident_batch_variants(collision, sigma_model):
    cases = [W.random_drop(nx, ny, seed=nx, wall_y=1, rho_ratio=10.0, gravity=1e-6,
                           collision=collision, sigma_model=sigma_model, beta=0.4, psi0=0.2,
                           gradpsi_x=1e-3) for nx, ny in ((75, 66), (130, 200), (65, 40))]
    outs = []
    for resident in (True, False):
        with lbm.Batch(cases, precision="fp32") as b:
            b.init_all()
            if not resident:
                lbm.lbm_batch_set_persistent(b.b, 0)
            b.step(33).step(40)
            outs.append([b.populations(i) for i in range(len(cases))])
    for (ga, fa), (gb, fb) in zip(*outs):
        assert np.array_equal(ga, gb) and np.array_equal(fa, fb)


@pytest.mark.parametrize("n", [2, 7, 30, 45])
def test_resident_batches_of_a_few_waves(n):
    """Counts for which the waves' blocks stay below the tallest that fit (30, 45) or not."""
    rng = np.random.default_rng(n)
    cases = [W.random_drop(int(rng.integers(32, 257)), int(rng.integers(32, 257)), seed=i,
                           rho_ratio=100.0) for i in range(n)]
    outs = []
    for resident in (True, False):
        with lbm.Batch(cases, precision="fp32") as b:
            b.init_all()
            if not resident:
                lbm.lbm_batch_set_persistent(b.b, 0)
            b.step(33)
            outs.append([b.populations(i) for i in range(n)])
    for (ga, fa), (gb, fb) in zip(*outs):
        assert np.array_equal(ga, gb) and np.array_equal(fa, fb)


def test_grids_beyond_shared_memory_and_of_one_node_take_the_other_forms():
    for nx, ny in ((1, 30), (30, 1), (700, 900)):
        case = W.random_drop(nx, ny, seed=4, wall_y=1, rho_ratio=10.0)
        with lbm.Simulation(case, precision="fp32") as sim:
            sim.init_case()
            before = lbm.lbm_state_device(sim.ctx)[0]
            sim.step(17)
            assert lbm.lbm_state_device(sim.ctx)[0] != before


def test_run_paths_name_the_form_that_runs_take():
    """lbm_get_run_path against where a run leaves the state (in place: resident), for run lengths,
    after each setting that keeps runs from the resident kernel and after lbm_set_resident."""
    case = W.random_drop(70, 60, seed=9, rho_ratio=10.0)
    with lbm.Simulation(case, precision="fp32") as sim:
        sim.init_case()

        def check(n, resident, launches=None):
            path, count = lbm.lbm_get_run_path(sim.ctx, n)
            before = lbm.lbm_state_device(sim.ctx)[0]
            sim.step(n)
            assert (lbm.lbm_state_device(sim.ctx)[0] == before) == resident
            assert (path == lbm.LBM_PATH_RESIDENT) == resident
            assert launches is None or count == launches

        check(17, True, 1)
        check(15, False, 15)
        check(1, False, 1)
        for keep, back in ((lambda: lbm.lbm_set_persistent(sim.ctx, 0), None),
                           (lambda: lbm.lbm_set_launch(sim.ctx, 4, 0), None),
                           (lambda: lbm.lbm_set_resident(sim.ctx, 0), None),
                           (lambda: lbm.lbm_set_graphs(sim.ctx, 0),
                            lambda: lbm.lbm_set_graphs(sim.ctx, 1))):
            keep()
            check(17, False, 17)
            if back:
                back()
            lbm.lbm_set_resident(sim.ctx, 1)
            check(17, True, 1)
        lbm.lbm_set_persistent(sim.ctx, 1)
        assert lbm.lbm_get_run_path(sim.ctx, 17) == (lbm.LBM_PATH_MULTI, 1)
        for bad in (0, -3):
            with pytest.raises(lbm.LbmError):
                lbm.lbm_get_run_path(sim.ctx, bad)
        for bad in (3, -1):
            with pytest.raises(lbm.LbmError):
                lbm.lbm_set_resident(sim.ctx, bad)
    flow = W.shear_circle(L0=64, u0=0.03)
    flow.update(reverse_step=20)
    with lbm.Simulation(flow, precision="fp32") as sim:   # 20 steps, then 20 in the other direction
        sim.init_case()
        assert lbm.lbm_get_run_path(sim.ctx, 40) == (lbm.LBM_PATH_RESIDENT, 2)
        assert lbm.lbm_get_run_path(sim.ctx, 25) == (lbm.LBM_PATH_RESIDENT, 1 + 5)


def test_run_paths_of_a_batch():
    cases = W.ensemble(6)
    with lbm.Batch(cases, precision="fp32") as b:
        b.init_all()
        path, waves = lbm.lbm_batch_get_run_path(b.b, 40)
        assert path == lbm.LBM_PATH_RESIDENT and 1 <= waves <= 6
        assert lbm.lbm_batch_get_run_path(b.b, 15) == (lbm.LBM_PATH_GRAPHS, 15)
        assert lbm.lbm_batch_get_run_path(b.b, 1) == (lbm.LBM_PATH_SINGLE, 1)
        for keep in (lambda: lbm.lbm_batch_set_persistent(b.b, 0),
                     lambda: lbm.lbm_batch_set_launch(b.b, 8, 0),
                     lambda: lbm.lbm_batch_set_resident(b.b, 0)):
            keep()
            assert lbm.lbm_batch_get_run_path(b.b, 40) == (lbm.LBM_PATH_GRAPHS, 40)
            lbm.lbm_batch_set_resident(b.b, 1)
            assert lbm.lbm_batch_get_run_path(b.b, 40) == (path, waves)
        lbm.lbm_batch_set_persistent(b.b, 1)
        assert lbm.lbm_batch_get_run_path(b.b, 40) == (lbm.LBM_PATH_MULTI, 1)
        with pytest.raises(lbm.LbmError):
            lbm.lbm_batch_get_run_path(b.b, 0)
        with pytest.raises(lbm.LbmError):
            lbm.lbm_batch_set_resident(b.b, 2)


def test_a_failed_tuning_leaves_the_resident_kernel_on():
    """Tuning fails where it may not wait for the batch's stream: during a capture of it."""
    import torch
    stream = torch.cuda.Stream()
    with lbm.Batch(W.ensemble(3), precision="fp32", stream=stream.cuda_stream) as b:
        b.init_all()
        assert lbm.lbm_batch_get_run_path(b.b, 40)[0] == lbm.LBM_PATH_RESIDENT
        torch.cuda.synchronize()
        with pytest.raises(Exception):
            with torch.cuda.graph(torch.cuda.CUDAGraph(), stream=stream,
                                  capture_error_mode="relaxed"):
                try:
                    lbm.lbm_batch_tune(b.b, 2)
                    failed = False
                except lbm.LbmError:
                    failed = True
        assert failed
        assert lbm.lbm_batch_get_run_path(b.b, 40)[0] == lbm.LBM_PATH_RESIDENT


def test_contexts_on_streams_of_their_own():
    """Contexts side by side on five streams, four with a part of the device and one in the other
    forms, over more than one launch's steps, against the whole device and against one launch per step on the default stream."""
    import torch
    shapes = ((64, 64, "fp32"), (130, 128, "fp32"), (200, 200, "bf16"), (161, 481, "fp32"),
              (256, 256, "bf16"))
    streams = [torch.cuda.Stream() for _ in shapes]
    cases = [W.random_drop(nx, ny, seed=nx, wall_x=1, wall_y=2, rho_ratio=10.0) for nx, ny, _ in shapes]

    def state(sim):
        raw = sim.save_state()[0]
        sim.close()
        return raw

    sims = [lbm.Simulation(c, precision=p, stream=s.cuda_stream)
            for c, (_, _, p), s in zip(cases, shapes, streams)]
    for sim in sims:
        sim.init_case()
        assert lbm.lbm_get_run_path(sim.ctx, 4120) == (
            (lbm.LBM_PATH_GRAPHS, 4120) if sim.nx == 200 else (lbm.LBM_PATH_RESIDENT, 2))
    for sim in sims:
        sim.step(4120)
    got = [state(sim) for sim in sims]
    for i, (c, (_, _, p)) in enumerate(zip(cases, shapes)):
        one = lbm.Simulation(c, precision=p).init_case()
        lbm.lbm_set_resident(one.ctx, 0)
        assert np.array_equal(got[i], state(one.step(4120)))
        alone = lbm.Simulation(c, precision=p, stream=streams[i].cuda_stream).init_case().step(2000)
        lbm.lbm_set_resident(alone.ctx, 2)     # another split for the rest of the run
        alone.step(1100)
        lbm.lbm_set_resident(alone.ctx, 1)
        assert np.array_equal(got[i], state(alone.step(1020)))


def test_a_grid_that_shares_the_device_better_in_the_other_forms():
    import torch
    case = W.random_drop(512, 256, seed=3, rho_ratio=10.0)
    stream = torch.cuda.Stream()
    with lbm.Simulation(case, precision="bf16", stream=stream.cuda_stream) as sim, \
            lbm.Simulation(case, precision="bf16") as default:
        assert lbm.lbm_get_run_path(sim.ctx, 40)[0] == lbm.LBM_PATH_GRAPHS
        lbm.lbm_set_resident(sim.ctx, 2)
        assert lbm.lbm_get_run_path(sim.ctx, 40)[0] == lbm.LBM_PATH_RESIDENT
        assert lbm.lbm_get_run_path(default.ctx, 40)[0] == lbm.LBM_PATH_RESIDENT


@pytest.mark.parametrize("form", ["fp32", "half rows", "bf16", "flow"])
def test_waits_for_messages_run_out_and_are_reported(form):
    """The waits for the neighbouring blocks are bounded: where no messages come (none is sent), every
    block gives up after its first step and the run reports LBM_ERR_TIMEOUT; initialising the state
    again clears it, and the same mailboxes then serve a run like a fresh context's."""
    case = (W.shear_circle(L0=130, u0=0.03) if form == "flow" else
            W.random_drop(70, 60, seed=7, wall_y=1, rho_ratio=100.0) if form == "half rows" else
            W.random_drop(200, 700, seed=7, wall_x=1, rho_ratio=100.0))
    precision = "bf16" if form == "bf16" else "fp32"
    with lbm.Simulation(case, precision=precision) as a, \
            lbm.Simulation(case, precision=precision) as fresh:
        a.init_case().step(20)
        lbm.lbm_check(a.ctx)
        lbm.lbm_inject_timeout(a.ctx, 2)
        assert lbm.lbm_get_run_path(a.ctx, 40)[0] == lbm.LBM_PATH_RESIDENT
        a.step(40)
        for read in (lambda: lbm.lbm_check(a.ctx), a.fields, a.save_state):
            with pytest.raises(lbm.LbmError) as e:
                read()
            assert e.value.status == lbm.LBM_ERR_TIMEOUT
        lbm.lbm_inject_timeout(a.ctx, 0)
        a.init_case().step(37)
        lbm.lbm_check(a.ctx)
        fresh.init_case().step(37)
        assert np.array_equal(a.save_state()[0], fresh.save_state()[0])
