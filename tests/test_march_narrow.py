"""CTAs of 64 and 32 threads of the row march (narrow strips): the rule that picks them, and their states against the tile
kernel and against 128-thread CTAs, bitwise."""
import dataclasses

import numpy as np
import pytest

import workloads as W
from test_host_runtime import fake, library, run, simulation   # noqa: F401 (fixture)

# blocks of 32 columns that a staged row has room for
SLOTS = {128: {(0, 0): 10, (0, 1): 9, (1, 0): 10, (1, 1): 9}, 64: {(0, 0): 5, (0, 1): 4, (1, 0): 6, (1, 1): 6},
         32: {(0, 0): 2, (0, 1): 2, (1, 0): 2, (1, 1): 2}}
FIELDS = ("phi", "rho", "ux", "uy", "p")


@pytest.fixture(scope="module")
def lbm():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1110_5004_gb300 import build
    build.build()
    import paper_1110_5004_gb300 as m
    return m


def launched_shapes(widths, storage, s_form):
    lbm, f, events = library()
    seen = {}
    for nx in widths:
        ny = 3000 if nx <= 1200 else 9
        s = simulation(lbm, nx, ny, storage, s_form)
        s.set_kernel(lbm.LBM_KERNEL_ROWS)
        s.set_tile(0, ny)                                   # one segment: as many CTAs as strips
        f.fake_clear()
        s.step(1)
        (e,) = events()
        assert e.what == b"k_march"
        threads, strips = e.n % 1024, e.n // 1024
        w = -(-nx // (2 * strips))
        assert w <= threads - 6, (nx, threads, strips)
        blocks = -(-nx // 32)
        for k in range(strips):
            need = blocks
            if nx >= 2 * w + 8:
                lo, hi = (2 * w * k - 4) % nx // 32, (2 * w * k + 2 * w + 3) % nx // 32
                wraps = (2 * w * k - 4) % nx > (2 * w * k + 2 * w + 3) % nx
                need = blocks - lo + hi + 1 if wraps else hi - lo + 1
            assert need <= SLOTS[threads][min(storage, 1), s_form], (nx, threads, strips, k, need)
        seen.setdefault(threads, []).append(nx)
        s.close()
    assert {32, 64, 128} <= set(seen)
    assert max(seen[32]) <= 52 and 52 in seen[32] and 116 in seen[64] and 128 in seen[128] and 244 in seen[128]
    short = simulation(lbm, 16, 16, storage, s_form)        # one row a segment with any: the widest
    short.set_kernel(lbm.LBM_KERNEL_ROWS)
    f.fake_clear()
    short.step(1)
    assert events()[0].n == 16 * 1024 + 128


@pytest.mark.parametrize("storage,s_form", [(0, 0), (0, 1), (1, 0), (2, 1)])
def test_every_strip_fits_its_cta(fake, storage, s_form):   # noqa: F811
    """Columns within the threads and staged blocks within the shared memory of the CTA that is launched, for every width
    to 1200 and some beyond."""
    run(fake, "launched_shapes", list(range(3, 1201)) + [2047, 2048, 4096, 14521, 73000], storage, s_form, module="test_march_narrow")


def workload(nx, ny, bcx, bcy, seed, rf=1, **phys):
    w = W.random_small(nx, ny, seed=seed, bc_x=bcx, bc_y=bcy, gravity=1e-5 if bcy == W.WALL else 0.0, remove_Fa=rf)
    return dataclasses.replace(w, phys=dataclasses.replace(w.phys, **phys))


@pytest.mark.gpu
@pytest.mark.parametrize("nx", [3, 4, 9, 26, 32, 51, 52, 53, 64, 77, 96, 115, 116, 117, 245, 250, 256, 267, 270, 271])
def test_narrow_strips_equal_tiles_bitwise(lbm, nx):
    """Both sides of each change of the thread count: step and moments, each wall combination and storage, segments of one
    row to the whole grid."""
    for k, (bcx, bcy, ny, st) in enumerate([(0, 0, 3005, 0), (1, 1, 3009, 0), (0, 1, 3012, 1), (1, 0, 3016, 2), (0, 0, 3007, 2),
                                            (1, 1, 3021, 1), (0, 1, 3033, 0)]):
        if nx < 4 and bcx:
            continue
        w = workload(nx, ny, bcx, bcy, seed=nx + k, rf=k & 1, ch_conservative=k == 2, fs_form=k % 3 == 0)
        want = lbm.Sim.from_workload(w, storage=st, kernel=lbm.LBM_KERNEL_TILES)
        want.step(8)
        want = want.checkpoint()
        for rows in (1, 4, ny, 0):
            s = lbm.Sim.from_workload(w, storage=st, kernel=lbm.LBM_KERNEL_ROWS)
            s.set_tile(0, rows)
            s.step(8)
            assert np.array_equal(s.checkpoint(), want), (k, rows)


def stacked(part, times):
    """The workload of `times` equal periodic boxes, one above the other."""
    tile = lambda a: np.ascontiguousarray(np.tile(np.asarray(a, np.float32), (times, 1)))
    return dataclasses.replace(part, ny=part.ny * times, phi0=tile(part.phi0), ux0=tile(part.ux0), uy0=tile(part.uy0), p0=tile(part.p0))


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny", [(30, 9000), (52, 6000), (100, 5000), (250, 4000), (268, 3500)])
def test_narrow_moments_equal_tiles_bitwise(lbm, nx, ny):
    """The march's moment pass (more than 2^18 cells): a periodic box of five equal parts has the tile kernel's fields of
    one part in each."""
    part, reps = workload(nx, ny // 5, 0, 0, seed=nx), 5
    assert part.nx * part.ny * reps > 1 << 18 >= part.nx * part.ny       # the march; the tile kernel
    for st in (0, 1):                                   # (BF16 rounding depends on the row)
        a = lbm.Sim.from_workload(part, storage=st, kernel=lbm.LBM_KERNEL_TILES)
        b = lbm.Sim.from_workload(stacked(part, reps), storage=st, kernel=lbm.LBM_KERNEL_ROWS)
        a.step(4)
        b.step(4)
        got, want = b.moments(), a.moments()
        assert all(np.array_equal(got[k], np.tile(want[k], (reps, 1))) for k in FIELDS), st


@pytest.mark.gpu
@pytest.mark.parametrize("forms", [dict(s_form=1), dict(f_form=1), dict(s_form=1, f_form=1)])
@pytest.mark.parametrize("nx", [5, 26, 52, 60, 116, 117, 250])
def test_march_only_forms_of_narrow_grids(lbm, nx, forms):
    """The forms that only the march runs: 200 equal boxes of 13 rows, a grid long enough for fewer threads, have the
    populations and fields of one, whose single rows take 128 (and are compared with the oracle elsewhere)."""
    for bcx in (W.PERIODIC, W.WALL):
        part, times = workload(nx, 13, bcx, 0, seed=nx, **forms), 200
        a = lbm.Sim.from_workload(part, kernel=lbm.LBM_KERNEL_ROWS)
        a.step(6)
        state = lambda s: s.checkpoint()[64:64 + s.ny * -(-nx // 32) * 32 * 76].reshape(s.ny, -1)
        want, fields = np.tile(state(a), (times, 1)), a.moments()
        for rows in (0, 1, 5):
            b = lbm.Sim.from_workload(stacked(part, times), kernel=lbm.LBM_KERNEL_ROWS)
            b.set_tile(0, rows)
            b.step(6)
            assert np.array_equal(state(b), want), rows
        got = b.moments()
        assert all(np.array_equal(got[k], np.tile(fields[k], (times, 1))) for k in FIELDS)


@pytest.mark.gpu
@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("widest,wide_too", [(52, False), (116, False), (116, True)])
def test_batches_of_narrow_members_equal_alone(lbm, storage, widest, wide_too):
    """Batches whose members are all narrow take 32 or 64 threads, with one wide member 128: each member's state is the one
    it has alone, in both forms of the mass defect."""
    ws = [workload(9 + (37 * i) % (widest - 8), 300 + (53 * i) % 260, i & 1, (i >> 1) & 1, seed=i, rf=1, s_form=(i >> 2) & 1)
          for i in range(70)]
    if wide_too:
        ws += [workload(1500, 1500, 0, 1, seed=99), workload(1500, 1500, 0, 1, seed=98, s_form=1)]
    batch = lbm.Batch()
    sims = [lbm.Sim.from_workload(w, storage=storage) for w in ws]
    slots = [batch.add(s) for s in sims]
    batch.step(5)
    for s, w, slot in zip(sims, ws, slots):
        batch.remove(slot)
        alone = lbm.Sim.from_workload(w, storage=storage, kernel=lbm.LBM_KERNEL_ROWS)
        alone.step(5)
        assert np.array_equal(s.checkpoint(), alone.checkpoint()), w.nx


def wide_members():
    import time
    lbm, f, events = library()
    sims = [simulation(lbm, nx, ny) for nx, ny in ((3000000, 3), (52, 600))]
    batch = lbm.Batch()
    for s in sims:
        batch.add(s)
    t0 = time.perf_counter()
    batch.step(1)
    assert time.perf_counter() - t0 < 2.0


def test_strips_of_very_wide_members_are_chosen_quickly(fake):   # noqa: F811
    """A batch tries each thread count for each member: by width, not strip by strip (9 s for this one)."""
    run(fake, "wide_members", module="test_march_narrow")
