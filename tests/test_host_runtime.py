"""Host code of the library on a CUDA runtime without a device (fake_cudart.c): which memory its kernels are given, and
what is copied.  Cases whose failure on a device would be an illegal access are shown here."""
import ctypes
import os
import shutil
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    from paper_1110_5004_gb300 import build
    build.build()
    so = str(tmp_path_factory.mktemp("fake") / "libfake_cudart.so")
    subprocess.run([shutil.which("gcc") or "cc", "-shared", "-fPIC", "-O1", "-o", so, os.path.join(HERE, "fake_cudart.c")],
                   check=True)
    return so


def run(fake, function, *args, module="test_host_runtime"):
    """`function` of a test module in a process of its own, on the fake runtime."""
    code = "import sys; sys.path[:0] = [%r, %r]; import %s as t; t.%s(*%r)" % (ROOT, HERE, module, function, args)
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, env=dict(os.environ, LD_PRELOAD=fake))
    assert r.returncode == 0, r.stdout + r.stderr


class Event(ctypes.Structure):
    _fields_ = [("what", ctypes.c_char * 64), ("a", ctypes.c_void_p), ("b", ctypes.c_void_p), ("n", ctypes.c_longlong), ("smem", ctypes.c_longlong)]


def library():
    import paper_1110_5004_gb300 as lbm
    f = ctypes.CDLL(None)
    f.fake_event.restype = ctypes.POINTER(Event)
    f.fake_range.argtypes = [ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int, ctypes.c_int]
    return lbm, f, lambda: [f.fake_event(i).contents for i in range(f.fake_events())]


def simulation(lbm, nx, ny, storage=0, s_form=0):
    p = lbm.lbm_params(beta=0.001875, kappa=0.015, phi_star=1.0, theta_M=0.1, tau_f=0.8, tau_g_A=0.8, tau_g_B=0.8, rho_A=1.0,
                       rho_B=0.1, storage=storage, s_form=s_form)
    return lbm.Sim(nx, ny, p)


def checkpoint_memory(storage, s_form, mtype, device, offset):
    """Which memory the reordering kernel gets for a checkpoint buffer of that kind."""
    import numpy as np
    lbm, f, events = library()
    s = simulation(lbm, 83, 29, storage, s_form)
    n = s.checkpoint_bytes
    raw = np.zeros(n + 512, np.uint8)
    at = (-raw.ctypes.data) % 256 + offset
    buf = raw[at:at + n]
    f.fake_range(buf.ctypes.data, n, mtype, device)
    lo, hi = buf.ctypes.data, buf.ctypes.data + n
    in_place = (mtype == 3 or (mtype == 2 and device == 0)) and lo % 4 == 0
    for move in (s.checkpoint, s.restore):
        f.fake_clear()
        move(buf)
        ev = events()
        given = [e for e in ev if e.what == b"k_reorder"]
        inside = [e for e in given if lo <= e.b < hi]
        assert given and len(inside) == (len(given) if in_place else 0), (move.__name__, [hex(e.b) for e in given])
        # every byte that the kernel does not move itself is copied, once
        ends = [e.a if move == s.checkpoint else e.b for e in ev if e.what == b"copy"]
        size = [e.n for e in ev if e.what == b"copy"]
        copied = sum(k for a, k in zip(ends, size) if lo <= a < hi)
        populations = 96 * 29 * (76 if storage == 0 else 38)
        on_device = mtype in (2, 3)
        assert copied == n - (populations if in_place else 0) - (0 if on_device else 64)   # (host: the header directly)
    assert bytes(buf[:4]) == b"LBMC"


@pytest.mark.parametrize("storage,s_form", [(0, 0), (1, 0), (0, 1)])
@pytest.mark.parametrize("mtype,device,offset", [
    (2, 0, 0), (2, 0, 4), (2, 0, 1), (3, 0, 0),   # this device's memory, on a word's boundary and off it; managed memory
    (2, 1, 0), (2, 1, 16), (2, 1, 1),     # another device's
    (1, 0, 0), (0, -2, 0)])               # page-locked and pageable host memory
def test_checkpoint_kernel_gets_only_memory_it_can_address(fake, storage, s_form, mtype, device, offset):
    run(fake, "checkpoint_memory", storage, s_form, mtype, device, offset)


def diagnostics_share():
    lbm, f, events = library()
    for ny in (8, 100, 152, 153, 304, 305, 500, 608, 609, 3000):
        s = simulation(lbm, 33, ny)
        f.fake_clear()
        s.diagnostics()
        (e,) = [e for e in events() if e.what == b"k_diag"]
        blocks = e.n // 1024
        share = -(-blocks // 152)
        assert blocks <= ny and share * (e.smem + 1024) <= 233472, (ny, blocks, e.smem)
        assert (share + 1) * (e.smem + 1024) > 233472, (ny, blocks, e.smem)
        s.close()


def test_diagnostics_blocks_spread_over_the_device(fake):
    """The diagnostics' blocks are placed while the moment pass still runs: no SM has room for more than its share."""
    run(fake, "diagnostics_share")
