"""The row march's bounded wait for its rows.  The host's hold_tile hook leaves one CTA without copies, so its wait runs
out after a short limit: the launch ends by itself, every call that reads the state says LBM_ERR_TIMEOUT, and a new state
(initial fields or a checkpoint) is sound again."""
import dataclasses
import time

import numpy as np
import pytest

import workloads as W

LIMIT_NS = 20_000_000


@pytest.fixture(scope="module")
def lbm():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1110_5004_gb300 import build
    build.build()
    import paper_1110_5004_gb300 as m
    return m


def workload(nx, ny, bcx=0, **phys):
    w = W.random_small(nx, ny, seed=nx, bc_x=bcx, bc_y=W.WALL, gravity=1e-5, remove_Fa=1)
    return dataclasses.replace(w, phys=dataclasses.replace(w.phys, **phys))


def fields(w):
    return [np.ascontiguousarray(a, np.float32) for a in (w.phi0, w.ux0, w.uy0, w.p0)]


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny,storage,bcx,s_form,rows,crowd", [
    (300, 90, 0, 0, 0, 0, False), (300, 90, 1, 1, 0, 30, False), (40, 200, 2, 0, 0, 1, False), (250, 60, 0, 1, 1, 60, False),
    (33, 4, 0, 0, 0, 0, True)])
def test_a_wait_that_runs_out_is_reported_and_forgotten(lbm, nx, ny, storage, bcx, s_form, rows, crowd):
    """First, single-row and last segments; crowd: a simulation without a page-locked record."""
    w = workload(nx, ny, bcx, s_form=s_form)
    others = [lbm.Sim.from_workload(W.random_small(12, 9, seed=4), init=False) for _ in range(512 if crowd else 0)]
    ref = lbm.Sim.from_workload(w, storage=storage, kernel=lbm.LBM_KERNEL_ROWS)
    ref.step(3)
    good = ref.checkpoint()
    ref.step(5)
    want = ref.checkpoint()
    s = lbm.Sim.from_workload(w, storage=storage, kernel=lbm.LBM_KERNEL_ROWS)
    s.set_tile(0, rows)

    def give_up():
        s.set_wait_limit(LIMIT_NS, hold_tile=0)
        t0 = time.perf_counter()
        s.step(2)
        s.set_wait_limit(1_000_000_000)
        return t0

    t0 = give_up()
    assert s.step_status() == lbm._lib.LBM_ERR_TIMEOUT
    assert time.perf_counter() - t0 < 2.0
    assert s.step_status() == 0                       # read once
    out = np.empty((5, ny, nx), np.float32)
    for call in (s.moments, s.checkpoint, s.diagnostics, s.interfacial_force, lambda: s.moments_packed(out)):
        give_up()
        with pytest.raises(lbm.LBMError) as e:
            call()
        assert e.value.code == lbm._lib.LBM_ERR_TIMEOUT
    for new_state, steps in ((lambda: s.restore(good), 5), (lambda: s.init_fields(*fields(w)), 8)):
        give_up()
        new_state()
        assert s.step_status() == 0                   # the old state's launch is forgotten
        s.step(steps)
        assert np.array_equal(s.checkpoint(), want)
    del others


@pytest.mark.gpu
def test_a_batch_goes_on_after_a_wait_that_ran_out(lbm):
    """One member's first tile is held: its CTA hands back the tiles that it takes from the counter, so that those members
    are reported too, the launch takes every tile once, and the next launches are sound."""
    import torch
    stream = torch.cuda.current_stream()
    ws = [workload(250 + 3 * i, 190 + i) for i in range(40)]
    batch = lbm.Batch(stream=stream)
    batch.set_tile(0, 20)
    sims = [lbm.Sim.from_workload(w, stream=stream) for w in ws]
    sims[0].set_wait_limit(LIMIT_NS, hold_tile=0)
    slots = [batch.add(s) for s in sims]
    batch.step(1)
    status = [s.step_status() for s in sims]
    assert status[0] == lbm._lib.LBM_ERR_TIMEOUT and 1 <= sum(c != 0 for c in status) <= 2
    batch.remove(slots[0])
    sims[0].set_wait_limit(1_000_000_000)
    batch.add(sims[0])
    for s, w in zip(sims, ws):
        s.init_fields(*fields(w))
    batch.step(18)
    assert all(s.step_status() == 0 for s in sims)
    for s, w, slot in zip(sims, ws, slots):
        alone = lbm.Sim.from_workload(w, kernel=lbm.LBM_KERNEL_ROWS)
        alone.step(18)
        batch.remove(slot)
        assert np.array_equal(s.checkpoint(), alone.checkpoint())


@pytest.mark.gpu
def test_a_short_limit_of_the_resident_kernel_leaves_the_march_its_own(lbm):
    """A limit of a nanosecond, as a resident simulation may set, is no reason for the march to give up sound rows."""
    w = workload(2100, 300)
    a = lbm.Sim.from_workload(w, kernel=lbm.LBM_KERNEL_ROWS)
    b = lbm.Sim.from_workload(w, kernel=lbm.LBM_KERNEL_ROWS)
    a.set_wait_limit(1)
    for _ in range(5):
        a.step(20)
        b.step(20)
        assert a.step_status() == 0
    assert np.array_equal(a.checkpoint(), b.checkpoint())
    assert np.array_equal(a.moments()["phi"], b.moments()["phi"])
