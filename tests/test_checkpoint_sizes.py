"""Checkpoints in pieces through the work planes: grids whose planes hold a block or less than a row of populations, odd
numbers of blocks, and several pieces."""
import dataclasses

import numpy as np
import pytest

import workloads as W
from test_host_runtime import fake, library, run, simulation   # noqa: F401 (fixture)

SIZES = [(3, 3), (32, 3), (33, 3), (100, 3), (500, 3), (97, 4), (64, 5), (31, 40), (161, 7), (300, 61), (1000, 33)]


def pieces(nx, ny, storage, s_form):
    lbm, f, events = library()
    s = simulation(lbm, nx, ny, storage, s_form)
    buf = np.zeros(s.checkpoint_bytes, np.uint8)
    lo = buf.ctypes.data
    pitch = -(-nx // 32) * 32
    populations = ny * pitch * (76 if storage == 0 else 38)
    room = 24 * ny * pitch + 96 * ny                     # six planes and twelve partials a row
    for move in (s.checkpoint, s.restore):
        f.fake_clear()
        move(buf)
        at, staged = lo + 64, set()
        for e in events():
            if e.what == b"copy":
                host, dev = (e.a, e.b) if move == s.checkpoint else (e.b, e.a)
                assert host == at and e.n > 0
                at += e.n
                if at <= lo + 64 + populations:
                    staged.add(dev)
                    assert e.n <= room
        assert at == lo + len(buf) and len(staged) == 1, (move.__name__, at - lo, staged)


@pytest.mark.parametrize("storage,s_form", [(0, 0), (0, 1), (1, 0)])
def test_pieces_cover_a_checkpoint_and_fit_the_planes(fake, storage, s_form):   # noqa: F811
    for nx, ny in SIZES:
        run(fake, "pieces", nx, ny, storage, s_form, module="test_checkpoint_sizes")


@pytest.mark.gpu
@pytest.mark.parametrize("storage,s_form", [(0, 0), (1, 0), (2, 0), (0, 1), (2, 1)])
def test_host_and_device_checkpoints_are_alike(storage, s_form):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1110_5004_gb300 as lbm
    for k, (nx, ny) in enumerate(SIZES):
        bcx, bcy = (k & 1, k >> 1 & 1) if min(nx, ny) > 3 else (0, 0)
        w = W.random_small(nx, ny, seed=k, bc_x=bcx, bc_y=bcy, remove_Fa=1)
        w = dataclasses.replace(w, phys=dataclasses.replace(w.phys, s_form=s_form))
        s = lbm.Sim.from_workload(w, storage=storage)
        s.step(5)
        host = s.checkpoint()
        dev = torch.zeros(host.nbytes, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        s.checkpoint(dev)
        assert np.array_equal(dev.cpu().numpy(), host), (nx, ny)
        s.step(4)
        want = s.checkpoint()
        for source in (host, dev):
            t = lbm.Sim.from_workload(w, storage=storage, init=False)
            t.restore(source)
            assert np.array_equal(t.checkpoint(), host), (nx, ny)
            t.step(4)
            assert np.array_equal(t.checkpoint(), want), (nx, ny)
