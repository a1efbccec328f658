"""The one-launch step loop of small systems against stream launches of the
grid kernels, which share its arithmetic: positions and velocities are the
same bits, and the counters the same numbers."""
import threading
import time

import numpy as np
import pytest

import paper_0911_5631_gb300 as md
from mdcheck import DT, RC, ensure_built, state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def _run(pos, vel, L, steps, skin, **kw):
    s = md.Simulation(L, pos.shape[0], RC, skin, DT, **kw)
    s.set_state(pos, vel)
    for k in steps:
        s.step(k)
    out = s.get_state() + (s.measure(), s.cells(), s.neighbor_pairs()[1])
    s.close()
    return out


# sizes around a block's atoms (32, 64, 128), the changes of block size (a
# block per SM of 152) and the largest system of the loop; hot states with a
# thin skin that rebuild every few steps, reorders at almost every rebuild;
# a state whose lists are longer than the lanes' registers and stages hold
@pytest.mark.parametrize("n,rho,T,skin,reorder", [
    (110, 0.8, 1.0, 0.3, 100), (129, 0.8, 2.0, 0.2, 3), (2048, 0.8, 1.0, 0.4, 100), (4864, 0.7, 2.0, 0.25, 10),
    (4865, 0.7, 1.0, 0.4, 0), (9729, 0.9, 1.5, 0.4, 20), (20011, 0.6, 1.0, 0.5, 100), (29184, 0.8, 1.0, 0.4, 25),
    (29185, 0.8, 1.0, 0.4, 25), (1500, 1.05, 2.0, 0.46, 30)])
def test_run_loop_matches_stream_launches(n, rho, T, skin, reorder):
    pos, vel, L = state(n, rho, T, 51, jitter=0.05)
    steps = [1, 2, 60, 33]
    a = _run(pos, vel, L, steps, skin, reorder_interval=reorder)
    b = _run(pos, vel, L, steps, skin, reorder_interval=reorder, use_graphs=False)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    for k in ("step", "rebuilds", "reorders", "list_entries", "max_neighbors", "max_occupancy", "ke", "pe", "virial"):
        assert a[2][k] == b[2][k], k
    assert np.array_equal(a[3], b[3]) and a[4] == b[4]
    assert a[2]["rebuilds"] >= 3


def test_run_loop_grows_its_lists_and_reports_errors():
    pos, vel, L = state(3000, 0.6, 2.0, 52, jitter=0.05)
    a = _run(pos, vel, L, [150], 0.4, nbr_capacity=12)
    b = _run(pos, vel, L, [150], 0.4)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    assert a[2]["nbr_capacity"] > 12 and a[2]["step"] == b[2]["step"] == 150
    # two atoms thrown at each other until the force leaves its range
    s = md.Simulation(L, 3000, RC, 0.4, DT)
    v2 = vel.copy()
    v2[:] *= 120.0
    s.set_state(pos, v2)
    with pytest.raises(md.MDError) as e:
        s.step(200)
    assert e.value.code == md.MD_EUNSTABLE
    # the handle starts again from a sound state
    s.set_state(pos, vel)
    s.step(150)
    p, v = s.get_state()
    s.close()
    assert np.array_equal(p, b[0]) and np.array_equal(v, b[1])


# the cell-list-only loop (8 lanes per atom, 16 atoms per block; the last size
# is beyond the resident blocks and runs as graphs), both forms
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("n,rho,T,reorder", [(17, 0.2, 1.0, 100), (500, 0.8, 1.0, 7), (2049, 1.0, 2.0, 20),
                                             (9000, 0.7, 1.0, 0), (30000, 0.8, 1.0, 25)])
def test_cells_only_loop_matches_stream_launches(n, rho, T, reorder, prec):
    pos, vel, L = state(n, rho, T, 53, jitter=0.05)
    steps = [1, 2, 40, 23]
    out = []
    for graphs in (True, False):
        s = md.Simulation(L, n, RC, 0.0, DT, precision=prec, cell_list_only=True, reorder_interval=reorder,
                          use_graphs=graphs)
        s.set_state(pos, vel)
        for k in steps:
            s.step(k)
        out.append(s.get_state() + (s.measure(), s.cells()))
        s.close()
    a, b = out
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]) and np.array_equal(a[3], b[3])
    for k in ("step", "rebuilds", "reorders", "max_occupancy", "ke", "pe", "virial"):
        assert a[2][k] == b[2][k], k
    assert a[2]["rebuilds"] == 1 + sum(steps)


def test_run_loops_beside_other_work_on_the_gpu():
    # loops of several handles and threads while an ensemble's persistent
    # launch holds every SM: whether a loop starts as a whole or gives way to
    # graphs, the results are those of a handle alone
    sizes = [600, 2048, 9000, 20000]
    states = [state(n, 0.8, 1.0, 54 + k, jitter=0.05) for k, n in enumerate(sizes)]
    alone = [_run(p, v, L, [40, 80], 0.4) for p, v, L in states]
    cells = [(n, state(n, 0.8, 1.0, 60, jitter=0.05)) for n in (700, 5000)]

    def cells_run(n, st):
        s = md.Simulation(st[2], n, RC, 0.0, DT, precision="fp64", cell_list_only=True)
        s.set_state(st[0], st[1])
        s.step(60)
        out = s.get_state()
        s.close()
        return out

    cells_alone = [cells_run(n, st) for n, st in cells]
    pos, vel, L = state(16384, 0.8, 1.0, 59, jitter=0.05)
    with md.Ensemble(2 << 30) as e:
        e.set_shape(1024, 0, 1, 1 << 20)
        ids = [e.add(pos, vel, L) for _ in range(160)]
        e.run(ids, [0] * len(ids))
        e.sync()
        e.run(ids, [300] * len(ids))  # some tens of milliseconds on every SM
        got, errors = {}, []

        def work(key, fn):
            try:
                got[key] = fn()
            except Exception as exc:  # reported below, in the test's own thread
                errors.append(exc)

        jobs = [threading.Thread(target=work, args=(k, lambda k=k: _run(*states[k], [40, 80], 0.4)))
                for k in range(len(sizes))]
        jobs += [threading.Thread(target=work, args=(10 + k, lambda k=k: cells_run(*cells[k])))
                 for k in range(len(cells))]
        for j in jobs:
            j.start()
        for j in jobs:
            j.join()
        e.sync()
    assert not errors, errors
    for k in range(len(sizes)):
        assert np.array_equal(got[k][0], alone[k][0]) and np.array_equal(got[k][1], alone[k][1]), sizes[k]
        assert got[k][2]["rebuilds"] == alone[k][2]["rebuilds"]
    for k in range(len(cells)):
        assert np.array_equal(got[10 + k][0], cells_alone[k][0]) and np.array_equal(got[10 + k][1], cells_alone[k][1])


@pytest.mark.parametrize("kw", [dict(), dict(cell_list_only=True), dict(cell_list_only=True, precision="fp64")])
def test_a_barrier_that_runs_out_ends_the_loop(kw):
    # the first barrier of a loop never fills: of a rebuild (the state is hot:
    # its atoms have moved skin/2 when the loop starts; cells only, every step)
    n = 500
    pos, vel, L = state(n, 0.8, 1.0, 55, jitter=0.05)
    skin = 0.0 if kw else 0.01
    s = md.Simulation(L, n, RC, skin, DT, **kw)
    s.set_state(pos, vel)
    md.md_debug_loop(s.h, md.MD_HOLD_BARRIER)
    t = time.perf_counter()
    with pytest.raises(md.MDError) as e:
        s.step(20)
    t = time.perf_counter() - t
    assert e.value.code == md.MD_ECUDA and "barrier" in str(e.value)
    assert t < 1.7 * _one_wait(L, n, pos, vel), t  # one wait, not one at each barrier of the rebuild
    assert md.md_debug_loop(s.h)[1] == 0
    s.set_state(pos, vel)
    s.step(20)
    p, v = s.get_state()
    assert md.md_debug_loop(s.h)[1] == 19
    s.close()
    b = md.Simulation(L, n, RC, skin, DT, use_graphs=False, **kw)
    b.set_state(pos, vel)
    b.step(20)
    assert all(np.array_equal(x, y) for x, y in zip((p, v), b.get_state()))
    b.close()


def _one_wait(L, n, pos, vel):
    # a step's own barrier, the only one that a loop with a good list meets
    s = md.Simulation(L, n, RC, 0.4, DT)
    s.set_state(pos, vel)
    md.md_debug_loop(s.h, md.MD_HOLD_BARRIER)
    t = time.perf_counter()
    with pytest.raises(md.MDError):
        s.step(3)
    t = time.perf_counter() - t
    s.close()
    return t


def test_a_loop_that_cannot_start_gives_way_to_graphs():
    n = 3000
    pos, vel, L = state(n, 0.8, 1.5, 56, jitter=0.05)
    ref = _run(pos, vel, L, [40] * 8 + [5000] + [40] * 8, 0.4, use_graphs=False)
    s = md.Simulation(L, n, RC, 0.4, DT)
    s.set_state(pos, vel)
    md.md_debug_loop(s.h, md.MD_HOLD_GATE)
    for _ in range(8):
        s.step(40)
    # the first, third and sixth call tried; no step ran in a loop
    assert md.md_debug_loop(s.h, md.MD_HOLD_GATE) == (3, 0, 3)
    s.step(5000)  # (a call that takes graphs at once: the fourth after the sixth is the next to try)
    assert md.md_debug_loop(s.h, 0) == (3, 0, 3)
    for _ in range(8):
        s.step(40)
    launched, steps, shut = md.md_debug_loop(s.h)
    assert shut == 3 and steps == 39 * (launched - 3) == 39 * 7
    assert all(np.array_equal(x, y) for x, y in zip(s.get_state(), ref[:2]))
    # a call of three loops waits at the first one's gate only
    md.md_debug_loop(s.h, md.MD_HOLD_GATE)
    s.step(5000)
    assert md.md_debug_loop(s.h) == (launched + 3, steps, 4)
    s.close()


def test_many_large_loops_at_once_give_way_to_graphs():
    # four loops of two thirds of the device each: calls that overlap take
    # graphs, a handle alone its loops again after a while
    n, k, calls = 20011, 100, 12
    pos, vel, L = state(n, 0.8, 1.0, 57, jitter=0.05)
    sims = [md.Simulation(L, n, RC, 0.4, DT) for _ in range(4)]
    for s in sims:
        s.set_state(pos, vel)
    start = threading.Barrier(len(sims))

    def work(s):
        start.wait()
        for _ in range(calls):
            s.step(k)

    threads = [threading.Thread(target=work, args=(s,)) for s in sims]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    launched = [md.md_debug_loop(s.h)[0] for s in sims]
    assert sum(launched) < len(sims) * calls, launched
    for _ in range(20):
        sims[0].step(1 + k // 10)
    assert md.md_debug_loop(sims[0].h)[0] > launched[0]
    for _ in range(20):
        sims[1].step(1 + k // 10)
    out = [s.get_state() for s in sims]
    assert all(np.array_equal(x, y) for x, y in zip(out[0], out[1]))
    assert all(np.array_equal(x, y) for x, y in zip(out[2], out[3]))
    for s in sims:
        s.close()
    ref = _run(pos, vel, L, [k] * calls, 0.4, use_graphs=False)
    assert all(np.array_equal(x, y) for x, y in zip(out[2], ref[:2]))


# which calls run in loops, by the steps that ran in them: sizes up to the last
# that fits (about 12000 atoms without lists), the forms that have no loop
@pytest.mark.parametrize("n,kw,loops", [
    (29184, dict(), True), (29185, dict(), False), (500, dict(shell_bins=False), False),
    (500, dict(precision="fp64"), False), (500, dict(build="warp"), False), (500, dict(variant="list_rows"), False),
    (500, dict(use_graphs=False), False), (12000, dict(cell_list_only=True), True),
    (12000, dict(cell_list_only=True, precision="fp64"), True), (30000, dict(cell_list_only=True), False)])
def test_which_calls_run_in_loops(n, kw, loops):
    pos, vel, L = state(n, 0.8, 1.0, 58, jitter=0.05)
    s = md.Simulation(L, n, RC, 0.0 if "cell_list_only" in kw else 0.4, DT, **kw)
    s.set_state(pos, vel)
    for k in (1, 30, 2):
        s.step(k)
    assert md.md_debug_loop(s.h) == ((2, 30, 0) if loops else (0, 0, 0))
    s.set_profiling(True)
    s.step(3)
    assert md.md_debug_loop(s.h)[0] == (2 if loops else 0)
    s.close()
