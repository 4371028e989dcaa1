"""The step, moment, diagnostic and transfer routes at the sizes where their rules and tiles change: each against
another route of the same arithmetic bitwise, the FP64 oracle, or a plain FP64 restatement."""
import ctypes
import dataclasses
import threading

import numpy as np
import pytest

import oracle
import workloads as W

TOL = 1e-5                 # of the FP64 oracle, FP32 storage
MARCH_W, MARCH_W_DIRECT = 122, 109   # widest half strip of the row march (and with s_form 1)
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


def workload(nx, ny, bcx, bcy, seed, rf=1, **phys):
    w = W.random_small(nx, ny, seed=seed, bc_x=bcx, bc_y=bcy, gravity=1e-5 if bcy == W.WALL else 0.0, remove_Fa=rf)
    return dataclasses.replace(w, phys=dataclasses.replace(w.phys, **phys))


# ---- the columns a strip stages ----------------------------------------------------------------
@pytest.mark.parametrize("w_max,slots", [(MARCH_W, 10), (MARCH_W_DIRECT, 9)])
def test_staged_blocks_cover_every_column_a_strip_reads(w_max, slots):
    """Host restatement of a strip's staged blocks (of 32 columns): within the shared-memory slots, inside the row, and
    covering the columns of both halves with their pull and ghost columns, for every width to 1100 and some
    beyond."""
    for nx in list(range(3, 1101)) + [2047, 2048, 2049, 3193, 4096, 14521]:
        strips = (nx + 2 * w_max - 1) // (2 * w_max)
        w = (nx + 2 * strips - 1) // (2 * strips)
        blocks = (nx + 31) // 32
        for strip in range(strips):
            x0 = strip * 2 * w
            b0, run1, run2 = 0, blocks, 0
            if nx >= 2 * w + 8:
                xs, xe = (x0 - 4) % nx, (x0 + 2 * w + 3) % nx
                b0 = xs >> 5
                run1, run2 = ((xe >> 5) - b0 + 1, 0) if xs <= xe else (blocks - b0, (xe >> 5) + 1)
            assert run1 + run2 <= slots and b0 + run1 <= blocks and run2 <= blocks, (nx, strip)
            staged = [b0 + k for k in range(run1)] + list(range(run2))
            for x in range(x0 - 4, x0 + 2 * w + 4):
                b = (x % nx) >> 5
                slot = b - b0 if b >= b0 else run1 + b
                assert staged[slot] == b, (nx, strip, x)


# ---- row march against tile kernel and oracle --------------------------------------------------
@pytest.mark.gpu
@pytest.mark.parametrize("nx", [4, 5, 31, 32, 33, 65, 2 * MARCH_W - 1, 2 * MARCH_W, 2 * MARCH_W + 1, 2 * MARCH_W + 8,
                                4 * MARCH_W, 4 * MARCH_W + 1, 516])
def test_march_strips_equal_tiles_bitwise(lbm, nx):
    """Widths around one, two and three strips, grids of few rows, each wall combination and storage, segments of one
    row to the whole grid: the state after 9 steps is the tile kernel's, bitwise."""
    for k, (bcx, bcy, ny, st) in enumerate([(0, 0, 3, 0), (1, 1, 4, 0), (0, 1, 11, 1), (1, 0, 8, 2), (0, 0, 17, 2),
                                            (1, 1, 23, 1), (0, 1, 14, 0)]):
        w = workload(nx, ny, bcx, bcy, seed=nx + k, rf=k & 1, ch_conservative=k == 2, fs_form=k % 3 == 0)
        want = lbm.Sim.from_workload(w, storage=st, kernel=lbm.LBM_KERNEL_TILES)
        want.step(9)
        want = want.checkpoint()
        for rows in (1, 2, 6, 0):
            s = lbm.Sim.from_workload(w, storage=st, kernel=lbm.LBM_KERNEL_ROWS)
            s.set_tile(0, rows)
            s.step(9)
            assert np.array_equal(s.checkpoint(), want), (k, rows)


@pytest.mark.gpu
@pytest.mark.parametrize("form", ["s_form", "f_form"])
@pytest.mark.parametrize("nx", [5, 33, 2 * MARCH_W_DIRECT, 2 * MARCH_W_DIRECT + 1, 2 * MARCH_W, 4 * MARCH_W_DIRECT + 3])
def test_march_only_forms_match_oracle(lbm, nx, form):
    """The direct mass defect and the forced order-parameter form run in the march alone: against the oracle, and every
    segment height alike."""
    for bcx, bcy in [(W.PERIODIC, W.WALL), (W.WALL, W.PERIODIC)]:
        w = workload(nx, 13, bcx, bcy, seed=nx, **{form: 1})
        ref = oracle.run(w, steps=10).moments()
        states = []
        for rows in (0, 1, 5):
            s = lbm.Sim.from_workload(w)
            s.set_tile(0, rows)
            s.step(10)
            states.append(s.checkpoint())
        assert all(np.array_equal(c, states[0]) for c in states)
        got = s.moments()
        u_den = max(np.abs(ref["ux"]).max(), np.abs(ref["uy"]).max(), w.phys.sigma / (w.phys.rho_A * w.phys.nu_A))
        for k in FIELDS:
            den = u_den if k in ("ux", "uy") else np.abs(ref[k]).max()
            assert np.abs(got[k] - ref[k]).max() <= TOL * den, (k, bcx, bcy)


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny", [(2000, 165), (2000, 198), (2000, 197), (2000, 196), (2000, 190), (2100, 520), (4900, 77),
                                   (40, 3200), (73000, 9)])
def test_segment_heights_at_y_walls(lbm, nx, ny):
    """Automatic heights from one row to the whole grid, with wall rows in any iteration of a segment and of its
    neighbours, and 20 rows by choice, against 5 rows everywhere: step and moments, bitwise."""
    for st, sform in [(0, 0), (1, 0), (2, 0), (0, 1)]:
        w = workload(nx, ny, (nx + st) & 1, W.WALL, seed=ny + st, s_form=sform)
        out = []
        for rows in (0, 5, 20):
            s = lbm.Sim.from_workload(w, storage=st, kernel=lbm.LBM_KERNEL_ROWS)
            s.set_tile(0, rows)
            s.step(4)
            out.append((s.checkpoint(), s.moments()))
        for state, m in out[1:]:
            assert np.array_equal(out[0][0], state), (st, sform)
            assert all(np.array_equal(out[0][1][k], m[k]) for k in FIELDS), (st, sform)


# ---- tile kernel: two tiles per CTA ------------------------------------------------------------
@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny,why", [
    (150, 450, "285 pairs: one wave of two per SM"), (256, 256, "256 pairs"), (38, 1500, "376 pairs, narrowest width"),
    (37, 1600, "too narrow for pairs"), (4000, 14, "fewest rows"), (4000, 13, "too few rows"),
    (256, 512, "just over one wave: single tiles"), (255, 561, "568 pairs: past the tail"), (257, 1021, "ragged")])
def test_paired_tiles_equal_row_march(lbm, nx, ny, why):
    for bcx, bcy, st in [(0, 1, 0), (0, 0, 1), (0, 1, 2), (0, 0, 0), (1, 1, 0)]:
        w = workload(nx, ny, bcx, bcy, seed=nx + st, rf=st != 1, ch_conservative=st == 2, fs_form=st == 1)
        a = lbm.Sim.from_workload(w, storage=st, kernel=lbm.LBM_KERNEL_TILES)
        b = lbm.Sim.from_workload(w, storage=st, kernel=lbm.LBM_KERNEL_ROWS)
        a.step(7)
        b.step(7)
        assert np.array_equal(a.checkpoint(), b.checkpoint()), (bcx, bcy, st)


# ---- batches -----------------------------------------------------------------------------------
@pytest.mark.gpu
@pytest.mark.parametrize("members", [3, 60])
def test_batch_rows_chosen_by_rounds_equal_alone(lbm, members):
    """Automatic tile heights of a few members (one round) and of many (several rounds), storages mixed."""
    ws = [workload(20 + (37 * i) % 290, 15 + (53 * i) % 260, i & 1, (i >> 1) & 1, seed=i, rf=i & 1) for i in range(members)]
    batch = lbm.Batch()
    sims = [lbm.Sim.from_workload(w, storage=i % 3) for i, w in enumerate(ws)]
    slots = [batch.add(s) for s in sims]
    batch.step(11)
    for i, (w, slot) in enumerate(zip(ws, slots)):
        batch.remove(slot)
        alone = lbm.Sim.from_workload(w, storage=i % 3, kernel=lbm.LBM_KERNEL_ROWS)
        alone.step(11)
        assert np.array_equal(sims[i].checkpoint(), alone.checkpoint()), i


# ---- diagnostics -------------------------------------------------------------------------------
def reduce_fp64(f, phs):
    """The record from the FP32 fields in FP64, and a bound on what another order of the sums may differ by: each side
    rounds at most n times, so 2 n 2^-53 of the sum of magnitudes, doubled for the rounding of the terms."""
    ph, u, v, p = (f[k].astype(np.float64) for k in ("phi", "ux", "uy", "p"))
    ny, nx = ph.shape
    c = np.clip((ph + phs) / (2.0 * phs), 0.0, 1.0)
    y, x = np.mgrid[0:ny, 0:nx].astype(np.float64)
    liq, gas = ph > 0.9 * phs, ph < -0.9 * phs
    eps = 4 * ph.size * 2.0 ** -53
    total = {k: (t.sum(), eps * np.abs(t).sum()) for k, t in
             dict(phi=ph, c=c, cx=c * x, cy=c * y, cu=c * u, cv=c * v, pl=p * liq, pg=p * gas).items()}
    out = {"sum_phi": total["phi"], "liquid_area": total["c"],
           "spread_radius": (0.5 * c.sum(axis=1).max(), 0.5 * eps * c.sum(axis=1).max()),
           "max_u": (np.sqrt(u * u + v * v).max(), 4 * 2.0 ** -53 * np.sqrt(u * u + v * v).max())}

    def quotient(num, den):
        (a, ea), (b, eb) = num, den
        return (a / b, ea / b + abs(a) * eb / b ** 2 + 2.0 ** -52 * abs(a / b)) if b > 0 else (0.0, 0.0)

    for name, k in (("centroid_x", "cx"), ("centroid_y", "cy"), ("vel_x", "cu"), ("vel_y", "cv")):
        out[name] = quotient(total[k], total["c"])
    out["p_liquid"] = quotient(total["pl"], (liq.sum(), 0.0))
    out["p_gas"] = quotient(total["pg"], (gas.sum(), 0.0))
    return out


def diagnose(lbm, f, phs):
    import torch
    from paper_1110_5004_gb300 import _lib
    dev = {k: torch.from_numpy(f[k]).cuda() for k in ("phi", "ux", "uy", "p")}
    torch.cuda.synchronize()
    ny, nx = f["phi"].shape
    rec = _lib.lbm_diag()
    rc = lbm.lib().lbm_diagnostics_fields_noalloc(dev["phi"].data_ptr(), dev["ux"].data_ptr(), dev["uy"].data_ptr(),
                                                  dev["p"].data_ptr(), nx, ny, phs, 5, None, ctypes.byref(rec))
    return rc, rec.as_dict()


def random_fields(nx, ny, seed, phs):
    r = np.random.default_rng(seed)
    f = {"phi": phs * r.uniform(-1.1, 1.1, (ny, nx)), "ux": 0.01 * r.standard_normal((ny, nx)),
         "uy": 0.01 * r.standard_normal((ny, nx)), "p": 1e-3 * r.standard_normal((ny, nx))}
    f = {k: v.astype(np.float32) for k, v in f.items()}
    f["ux"].flat[::7] = 0.0
    f["uy"].flat[::5] = 1e-41             # subnormal
    f["phi"].flat[::3] = np.float32(phs)  # on the clamp
    f["phi"].flat[1::11] = np.float32(0.9 * phs)
    return f


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny,phs", [(1, 1, 1.0), (255, 3, 1.0), (257, 608, 0.7), (40, 609, 1.0), (300, 1217, 0.75),
                                       (33, 4256, 0.5), (31, 4865, 1.3), (70, 8192, 1.0), (2049, 5, 1.0)])
def test_diagnostics_equal_fp64_sums(lbm, nx, ny, phs):
    """One row per block to eight and a remainder, rows shorter and longer than a block, phi* that FP32 and powers of
    two represent or not, values on the phase limits, zeros and subnormals."""
    f = random_fields(nx, ny, nx + ny, phs)
    rc, got = diagnose(lbm, f, phs)
    assert rc == 0 and got["finite"] == 1 and got["step"] == 5
    for k, (want, bound) in reduce_fp64(f, phs).items():
        assert abs(got[k] - want) <= bound, (k, got[k], want, bound)


@pytest.mark.gpu
@pytest.mark.parametrize("field", ["phi", "ux", "uy"])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_one_bad_cell_is_reported_wherever_it_is(lbm, field, bad):
    """A value that is not finite in any thread's first, middle or last cell, or in any block, makes the record not
    finite, whatever follows it."""
    nx, ny = 520, 1300
    f = random_fields(nx, ny, 3, 1.0)
    for y, x in [(0, 0), (0, 300), (1, 519), (700, 255), (1299, 0), (1299, 519)]:
        keep = f[field][y, x]
        f[field][y, x] = bad
        rc, got = diagnose(lbm, f, 1.0)
        assert got["finite"] == 0, (y, x)
        f[field][y, x] = keep


@pytest.mark.gpu
def test_more_simulations_than_record_slots_and_threads(lbm):
    """Diagnostics of more simulations than the pool has page-locked records (the rest copy theirs), the same again
    once all were given back, and from several threads at once."""
    w = W.random_small(12, 9, seed=4)
    want = lbm.Sim.from_workload(w).diagnostics()
    for _ in range(2):
        sims = [lbm.Sim.from_workload(w) for _ in range(520)]
        assert all(s.diagnostics() == want for s in sims)
        del sims
    wrong = []

    def worker(seed):
        wk = W.random_small(40 + seed, 30, seed=seed)
        ref = None
        for _ in range(20):
            s = lbm.Sim.from_workload(wk)
            s.step(3)
            d = s.diagnostics()
            ref = ref or d
            if d != ref or d["step"] != 3:
                wrong.append((seed, d))

    threads = [threading.Thread(target=worker, args=(i,)) for i in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong


# ---- transfers ---------------------------------------------------------------------------------
@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny,kernel", [(33, 9, 0), (64, 20, 0), (45, 700, 0), (601, 437, 0), (530, 501, 0)])
def test_fields_in_place_at_any_alignment(lbm, nx, ny, kernel):
    """Initial fields read from, and moments and forces written to, device memory that starts at any float, alone or
    mixed with host arrays, on both sides of the small-grid rule: bitwise what host arrays give, and nothing written
    outside."""
    import torch
    w = workload(nx, ny, W.PERIODIC, W.WALL, seed=nx)
    src = {k: np.ascontiguousarray(getattr(w, k), np.float32) for k in ("phi0", "ux0", "uy0", "p0")}
    n, guard = nx * ny, 12345.0

    def on_device(a, off):
        b = torch.full((off + a.size + 5,), guard, device="cuda")
        b[off:off + a.size] = torch.from_numpy(a.reshape(-1)).cuda()
        return b, b[off:off + a.size]

    ref = lbm.Sim.from_workload(w)
    ref.step(3)
    want, fa, ck = ref.moments(), ref.interfacial_force(), ref.checkpoint()
    for off in (1, 2, 7):
        dev = {k: on_device(a, off + i) for i, (k, a) in enumerate(src.items())}
        torch.cuda.synchronize()
        for host in ((), ("ux0",), ("phi0", "p0")):
            s = lbm.Sim(nx, ny, lbm.params_from_physical(w.phys))
            s.init_fields(*[src[k] if k in host else dev[k][1] for k in src])
            s.step(3)
            assert np.array_equal(s.checkpoint(), ck), (off, host)
            for host_out in ((), ("rho",)):
                out = {k: on_device(np.full((ny, nx), 7.0, np.float32), off + i) for i, k in enumerate(FIELDS)}
                torch.cuda.synchronize()
                got = {k: np.empty((ny, nx), np.float32) if k in host_out else out[k][1] for k in FIELDS}
                s.moments(got)
                for k in FIELDS:
                    v = got[k] if k in host_out else got[k].cpu().numpy().reshape(ny, nx)
                    assert np.array_equal(v, want[k]), (off, host, host_out, k)
                    whole = out[k][0].cpu().numpy()
                    assert (np.delete(whole, np.s_[off + FIELDS.index(k):off + FIELDS.index(k) + n]) == guard).all()
        f2 = {k: on_device(np.zeros((ny, nx), np.float32), off)[1] for k in ("fax", "fay")}
        torch.cuda.synchronize()
        s.interfacial_force(f2)
        for k in f2:
            assert np.array_equal(f2[k].cpu().numpy().reshape(ny, nx), fa[k]), (off, k)


@pytest.mark.gpu
@pytest.mark.parametrize("storage,s_form", [(0, 0), (1, 0), (2, 0), (0, 1)])
def test_checkpoint_in_any_memory(lbm, storage, s_form):
    """Host memory, and device memory on a 16-byte boundary and off it: the same bytes, and each restores."""
    import torch
    w = workload(83, 29, W.PERIODIC, W.WALL, seed=5, s_form=s_form)
    a = lbm.Sim.from_workload(w, storage=storage)
    a.step(7)
    want = a.checkpoint()
    a.step(6)
    later = a.checkpoint()
    for off in (0, 16, 8, 1):
        b = lbm.Sim.from_workload(w, storage=storage)
        b.restore(want)
        buf = torch.zeros(off + want.nbytes, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        b.checkpoint(buf[off:])
        assert np.array_equal(buf[off:].cpu().numpy(), want), off
        c = lbm.Sim.from_workload(w, storage=storage, init=False)
        c.restore(buf[off:])
        c.step(6)
        assert np.array_equal(c.checkpoint(), later), off


@pytest.mark.gpu
@pytest.mark.parametrize("bc", [W.PERIODIC, W.WALL])
def test_checkpoint_holds_populations_by_their_source_cell(lbm, bc):
    """A checkpoint keeps a population at the cell that it leaves (the state itself, at the row that it reaches): the
    pull of an initial checkpoint, half-way bounce-back included, sums to phi0.  Bound: 32 roundings of the sum of
    magnitudes."""
    nx, ny = 45, 21
    w = workload(nx, ny, bc, bc, seed=9)
    payload = lbm.Sim.from_workload(w).checkpoint()[64:].view(np.float32).reshape(ny, 2, 19, 32)
    f = payload.transpose(2, 0, 1, 3).reshape(19, ny, 64)[:, :, :nx].astype(np.float64)
    f[0] += f[18]
    e = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
    y, x = np.mgrid[0:ny, 0:nx]
    total = np.zeros((ny, nx))
    size = np.zeros((ny, nx))
    for a, (ex, ey) in enumerate(e):
        xs, ys = x - ex, y - ey
        out = (xs < 0) | (xs >= nx) | (ys < 0) | (ys >= ny)
        pulled = f[a][ys % ny, xs % nx]
        if bc == W.WALL:
            pulled = np.where(out, f[e.index((-ex, -ey))], pulled)
        total += pulled
        size += np.abs(pulled)
    assert (np.abs(total - w.phi0) <= 32 * 2.0 ** -24 * size).all()


# ---- graphs ------------------------------------------------------------------------------------
@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny,kernel", [(64, 48, 2), (256, 256, 2), (300, 90, 1)])
def test_steps_captured_in_a_graph_equal_eager(lbm, nx, ny, kernel):
    """Two steps and the initialisation from device fields, recorded once and replayed."""
    import torch
    w = workload(nx, ny, W.PERIODIC, W.WALL, seed=2)
    stream = torch.cuda.Stream()
    s = lbm.Sim.from_workload(w, stream=stream, kernel=kernel)
    dev = [torch.from_numpy(np.ascontiguousarray(getattr(w, k), np.float32)).cuda() for k in ("phi0", "ux0", "uy0", "p0")]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        s.step(2)
    with torch.cuda.stream(stream):
        for _ in range(3):
            graph.replay()
    stream.synchronize()
    ref = lbm.Sim.from_workload(w, kernel=kernel)
    ref.step(6)
    got, want = s.moments(), ref.moments()
    assert all(np.array_equal(got[k], want[k]) for k in FIELDS)
    init = torch.cuda.CUDAGraph()
    with torch.cuda.graph(init, stream=stream):
        s.init_fields(*dev)
        s.step(2)
    with torch.cuda.stream(stream):
        init.replay()
    stream.synchronize()
    ref = lbm.Sim.from_workload(w, kernel=kernel)
    ref.step(2)
    got, want = s.moments(), ref.moments()
    assert all(np.array_equal(got[k], want[k]) for k in FIELDS)


@pytest.mark.gpu
def test_batch_steps_captured_in_a_graph_equal_eager(lbm):
    """Direct batch launches (fewer steps than the batch's own graph) recorded and replayed between eager ones: every
    launch finds its tile counter at zero.  More tiles than one wave, so that the counter hands some out."""
    import torch
    ws = [workload(250 + 3 * i, 190 + i, 0, W.WALL, seed=i) for i in range(40)]
    stream = torch.cuda.Stream()
    batch = lbm.Batch(stream=stream)
    batch.set_tile(0, 20)
    sims = [lbm.Sim.from_workload(w) for w in ws]
    slots = [batch.add(s) for s in sims]
    batch.step(2)                                     # builds the work list
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        batch.step(2)
    with torch.cuda.stream(stream):
        for _ in range(3):
            graph.replay()
    batch.step(4)
    for w, s, slot in zip(ws, sims, slots):
        batch.remove(slot)
        alone = lbm.Sim.from_workload(w, kernel=lbm.LBM_KERNEL_ROWS)
        alone.step(2 + 3 * 2 + 4)
        got, want = s.moments(), alone.moments()
        assert all(np.array_equal(got[k], want[k]) for k in FIELDS)
