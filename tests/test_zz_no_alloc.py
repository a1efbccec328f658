"""md_forces_noalloc: forces without any device allocation.

Some callers may not allocate device memory -- code running inside a memory
pool or budget it does not own, or on a path where cudaMalloc/cudaFree must
not run because they synchronise the whole device.  md_forces_noalloc serves
them with a fixed scratch area inside the library.  This test calls it
through the C ABI twice in a row (the second call reuses the scratch the
first one left behind, at the maximum size) and compares each result with
the handle-based entry points (md_set_state + md_get_forces + md_measure,
FP64 form) and with the FP64 oracle, within the FP64 force tolerance used
throughout the tests.  A non-finite position is reported as MD_EUNSTABLE.
It runs last so that a failure here leaves every other test already run.
"""
import numpy as np
import pytest

import oracle
import paper_0911_5631_gb300 as md
from mdcheck import FORCE_TOL, RC, ensure_built, face_state, oracle_grid, rel_rms, state

pytestmark = pytest.mark.gpu


def _reference(pos, vel, L):
    s = md.Simulation(L, pos.shape[0], RC, 0.4, 0.005, precision="fp64")
    s.set_state(pos, vel)
    f = s.forces()
    m = s.measure()
    s.close()
    return f, m["pe"], m["virial"]


def _noalloc(torch, pos, L):
    n = pos.shape[0]
    tp = torch.tensor(pos, dtype=torch.float64, device="cuda")
    tf = torch.full((n, 3), np.nan, dtype=torch.float64, device="cuda")
    te = torch.full((2,), np.nan, dtype=torch.float64, device="cuda")
    md.md_forces_noalloc(L, n, RC, tp.data_ptr(), tf.data_ptr(), te.data_ptr())
    torch.cuda.synchronize()
    e = te.cpu().numpy()
    return tf.cpu().numpy(), float(e[0]), float(e[1])


def test_forces_noalloc_matches_handle_path_twice():
    torch = pytest.importorskip("torch")
    ensure_built()
    cases = [
        state(2048, 0.8, 1.0, 11, jitter=0.1),
        # the largest accepted size, after a smaller call left its data behind
        state(md.MD_NOALLOC_MAX_ATOMS, 0.8, 1.0, 12, jitter=0.1),
    ]
    for pos, vel, L in cases:
        f_ref, pe_ref, w_ref = _reference(pos, vel, L)
        f, pe, w = _noalloc(torch, pos, L)
        assert np.all(np.isfinite(f))
        assert rel_rms(f, f_ref) <= FORCE_TOL["fp64"]
        assert pe == pytest.approx(pe_ref, rel=10 * FORCE_TOL["fp64"])
        assert w == pytest.approx(w_ref, rel=10 * FORCE_TOL["fp64"])
        # and the FP64 oracle's cell-list forces on the same configuration
        pw = oracle.wrap(pos, L)
        f_orc, u_orc, w_orc = oracle.forces_cells(pw, L, oracle_grid(L, RC), RC, 1.0)
        assert rel_rms(f, f_orc) <= FORCE_TOL["fp64"]
        assert pe == pytest.approx(u_orc, rel=10 * FORCE_TOL["fp64"])
        assert w == pytest.approx(w_orc, rel=10 * FORCE_TOL["fp64"])


def test_forces_noalloc_reports_non_finite_positions():
    torch = pytest.importorskip("torch")
    ensure_built()
    pos, vel, L = state(2048, 0.8, 1.0, 13, jitter=0.1)
    bad = pos.copy()
    bad[77, 1] = np.nan
    bad[1500, 2] = np.inf
    tp = torch.tensor(bad, dtype=torch.float64, device="cuda")
    tf = torch.zeros((2048, 3), dtype=torch.float64, device="cuda")
    te = torch.zeros(2, dtype=torch.float64, device="cuda")
    with pytest.raises(md.MDError) as e:
        md.md_forces_noalloc(L, 2048, RC, tp.data_ptr(), tf.data_ptr(), te.data_ptr())
    assert e.value.code == md.MD_EUNSTABLE
    # the flag does not stick: the next call on finite input succeeds
    f, pe, w = _noalloc(torch, pos, L)
    assert np.all(np.isfinite(f)) and np.isfinite(pe)


def test_forces_noalloc_rejects_sizes_beyond_the_scratch():
    torch = pytest.importorskip("torch")
    ensure_built()
    n = md.MD_NOALLOC_MAX_ATOMS + 1
    L = [45.0, 45.0, 45.0]
    tp = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
    tf = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
    te = torch.zeros(2, dtype=torch.float64, device="cuda")
    with pytest.raises(md.MDError) as e:
        md.md_forces_noalloc(L, n, RC, tp.data_ptr(), tf.data_ptr(), te.data_ptr())
    assert e.value.code == md.MD_EINVAL
    assert "MD_NOALLOC_MAX_ATOMS" in str(e.value)
    # too many cells for the scratch area
    with pytest.raises(md.MDError) as e:
        md.md_forces_noalloc([80.0, 80.0, 80.0], 100, RC, tp.data_ptr(), tf.data_ptr(), te.data_ptr())
    assert e.value.code == md.MD_EINVAL


# (n, rho, jitter, aspect): one atom, one block of 32 atoms and one more, the
# 3-cell grid (every cell at a periodic face), the largest size that one block
# bins and the next, a dense state whose atoms queue more pairs than the
# queue holds, an elongated box, more than one scan tile of cells.
@pytest.mark.parametrize("case", [(1, 0.02, 0.0, (1, 1, 1)), (32, 0.7, 0.1, (1, 1, 1)), (33, 0.7, 0.1, (1, 1, 1)),
                                  (4096, 0.9, 0.1, (1, 1, 1)), (4097, 0.9, 0.1, (1.0, 1.3, 0.8)),
                                  (500, 3.0, 0.02, (1, 1, 1)), (6000, 3.0, 0.02, (1, 1, 1)),
                                  (3000, 0.7, 0.15, (20.0, 1.0, 1.0)), (300, 0.1, 0.3, (1, 1, 1))])
def test_forces_noalloc_at_the_edges_of_its_kernels(case):
    torch = pytest.importorskip("torch")
    ensure_built()
    n, rho, jitter, aspect = case
    pos, vel, L = state(n, rho, 1.0, 21, jitter=jitter, aspect=aspect)
    pw = oracle.wrap(pos, L)
    f_ref, u_ref, w_ref = oracle.forces_cells(pw, L, oracle_grid(L, RC), RC, 1.0)
    f, u, w = _noalloc(torch, pos, L)
    # FP64 sums in another order: a few ulps of the largest pair force
    scale = max(np.abs(f_ref).max(), 1.0)
    assert np.abs(f - f_ref).max() <= 1e-12 * scale * max(1.0, n / 1000.0)
    assert u == pytest.approx(u_ref, rel=10 * FORCE_TOL["fp64"], abs=1e-12)
    assert w == pytest.approx(w_ref, rel=10 * FORCE_TOL["fp64"], abs=1e-12)


# atoms on and beside the faces and in the corners, in boxes whose half edges
# are short binary numbers: one block bins the first three (the third with the
# largest number of cells that it takes), five kernels the last, whose scratch
# then holds a larger call's atoms
@pytest.mark.parametrize("box", [(8.0, 10.0, 12.0), (9.1, 11.7, 10.9), (18.0, 18.0, 18.0), (20.0, 24.0, 20.0)])
def test_forces_noalloc_with_atoms_on_the_faces(box):
    torch = pytest.importorskip("torch")
    ensure_built()
    big, _, Lb = state(20000, 0.8, 1.0, 22, jitter=0.1)
    _noalloc(torch, big, Lb)
    pos, _, L = face_state(box, 1.12, 64)
    f_ref, u_ref, w_ref = oracle.forces_brute(oracle.wrap(pos, L), L, RC, 1.0)
    f, u, w = _noalloc(torch, pos, L)
    # separations within two ulps of L/2 (4e-15), a pair force's slope of up to
    # 400 per unit (r > 1.03), six pairs an atom: 1e-11, of forces of 5 to 9
    assert np.abs(f - f_ref).max() <= 1e-11 * np.abs(f_ref).max()
    assert u == pytest.approx(u_ref, rel=1e-11)
    assert w == pytest.approx(w_ref, rel=1e-11)
