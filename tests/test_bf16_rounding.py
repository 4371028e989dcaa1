"""The rounding of BF16 storage, value by value: an initial state in BF16 against the same populations in FP32 storage,
rounded here by integer arithmetic."""
import dataclasses

import numpy as np
import pytest

import workloads as W


def blocks(checkpoint, nx, ny, per_cell):
    """(ny, blocks, bytes of a block) of a checkpoint's populations."""
    nb = -(-nx // 32)
    return checkpoint[64:64 + ny * nb * 32 * per_cell].reshape(ny, nb, 32 * per_cell)


def fields(kind, ny, nx):
    """Initial fields whose populations meet the corners: subnormal values, halves between two BF16 numbers, the largest
    finite numbers and beyond, infinities and NaN."""
    r = np.random.default_rng(11)
    z = np.zeros((ny, nx), np.float32)
    phi = r.uniform(-1, 1, (ny, nx)).astype(np.float32)
    if kind == "ordinary":
        return phi, (0.1 * r.standard_normal((ny, nx))).astype(np.float32), z + np.float32(0.03), (1e-3 * r.standard_normal((ny, nx))).astype(np.float32)
    if kind == "every_exponent":
        p = r.integers(0, 1 << 32, (ny, nx), dtype=np.uint64).astype(np.uint32).view(np.float32).copy()
        return phi, z, z, p                                    # finite, subnormal, infinite and NaN bit patterns
    if kind == "largest":
        u = (1.0e18 * r.uniform(0.5, 4.0, (ny, nx))).astype(np.float32)
        return phi, u, z, z                                    # rho u^2 passes the largest finite number
    p = (np.float32(36.0) * r.integers(0, 1 << 23, (ny, nx)).astype(np.uint32).view(np.float32)).astype(np.float32)
    return phi, z, z, p                                        # "subnormal": w p below 2^-126


def nearest(bits):
    odd = (bits >> 16) & 1
    return ((bits.astype(np.uint64) + 0x7FFF + odd) >> 16).astype(np.uint16)


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["ordinary", "every_exponent", "largest", "subnormal"])
def test_bf16_bits_are_those_of_the_integer_formula(kind):
    """gbar: the value's bits plus 16 bits of a hash of them and of the cell's place in a checkpoint, cut off; infinities stay
    themselves.  f: to nearest, even.  A NaN is some NaN."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1110_5004_gb300 as lbm
    nx, ny = 417, 301
    phys = dataclasses.replace(W.random_small(8, 8, seed=1).phys, rho_A=1000.0, rho_B=1.0)
    f = fields(kind, ny, nx)
    raw = {}
    for st in (0, 2):
        s = lbm.Sim(nx, ny, lbm.params_from_physical(phys, st))
        s.init_fields(*f)
        raw[st] = blocks(s.checkpoint(), nx, ny, 76 if st == 0 else 38)
    want = np.ascontiguousarray(raw[0]).view(np.uint32).reshape(ny, -1, 19, 32)
    got = np.ascontiguousarray(raw[2][:, :, 128:]).view(np.uint16).reshape(ny, -1, 17, 32)
    nb = want.shape[1]
    y, b, lane = np.mgrid[0:ny, 0:nb, 0:32]
    real = b * 32 + lane < nx
    key = (y * (nb * 32 * 38) + b * (32 * 38) + lane * 2).astype(np.uint64)
    seen = set()
    for a in range(1, 18):
        bits, out = want[:, :, a], got[:, :, a - 1]
        special = (bits & 0x7F800000) == 0x7F800000
        nan = special & ((bits & 0x7FFFFF) != 0)
        expect = nearest(bits)
        if a >= 9:
            where = key + np.uint64(128 + (a - 1) * 64)
            hashed = ((bits.astype(np.uint64) ^ where) * np.uint64(0x9E3779B1)) & np.uint64(0xFFFFFFFF)
            stochastic = ((bits.astype(np.uint64) + (hashed >> np.uint64(16))) >> np.uint64(16)).astype(np.uint16)
            expect = np.where(special, (bits >> 16).astype(np.uint16), stochastic)
        ok = np.where(nan, ((out & 0x7F80) == 0x7F80) & ((out & 0x7F) != 0), out == expect) | ~real
        assert ok.all(), (a, [(hex(v), hex(g), hex(e)) for v, g, e in zip(bits[~ok][:4], out[~ok][:4], expect[~ok][:4])])
        exponent = (bits[real] >> 23) & 0xFF
        seen |= {k for k, m in (("nan", nan), ("inf", special & ~nan)) if (m & real).any()}
        seen |= {k for k, m in (("sub", exponent == 0), ("top", exponent == 254)) if m.any()}
    assert {"ordinary": set(), "every_exponent": {"nan", "sub"}, "largest": {"top", "inf"}, "subnormal": {"sub"}}[kind] <= seen
