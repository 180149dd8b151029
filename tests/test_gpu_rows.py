"""Row-per-lane codec core against the oracle, bit for bit: group and row
edges, deltas at the edges of the 8-, 16- and 32-bit paths, values near ties,
levels around the fast path's limit, unaligned inputs and outputs."""

import numpy as np
import pytest
import torch

import oracle
from paper_2308_05199_gb300 import workloads

pytestmark = pytest.mark.gpu

BLOCKS = [16, 32, 64, 128]
SIZES = [1, 31, 33, 1023, 1024, 1025, 2048, 3 * 1024 + 17, 9000, 70001]
EB = 0.5  # 2 eb = 1: levels are the values' nearest integers
KINDS = ["d8", "d16", "wide", "edge8", "edge16", "limit", "far", "ties", "offset", "mixed"]


@pytest.fixture(scope="session")
def zc():
    from paper_2308_05199_gb300 import build as zbuild, zc as z
    zbuild.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return z


def levels(kind, n, seed):
    r = np.random.Generator(np.random.PCG64(seed))
    if kind == "d8":
        return r.integers(-60, 60, n)
    if kind == "d16":
        return r.integers(-9000, 9000, n)
    if kind == "wide":
        return r.integers(-(1 << 19), 1 << 19, n)
    if kind == "edge8":  # deltas 127, -127, -128, 128 beside small ones
        return np.cumsum(r.choice([0, 1, -1, 127, -127, -128, 128], n, p=[.4, .2, .2, .05, .05, .05, .05])) % 8000
    if kind == "edge16":  # the largest deltas of the 16-bit path, and just beyond
        return r.choice([15999, -15999, 16000, -16000, 16001, 0, 5], n)
    if kind == "limit":
        return r.choice([0, 1, (1 << 22), -(1 << 22), (1 << 22) - 1, 1 << 21, -(1 << 21)], n)
    if kind == "far":  # both sides of 2^20
        return r.choice([1 << 20, (1 << 20) - 1, -(1 << 20), 1 - (1 << 20), 3, 1048000], n)
    if kind == "offset":
        return 300000 + r.integers(-100, 100, n)
    if kind == "mixed":
        q = r.integers(-3, 4, n)
        at = r.random(n) < 0.002
        return np.where(at, r.integers(-(1 << 21), 1 << 21, n), q)
    return r.integers(-200, 200, n)


def values(kind, n, seed, dtype):
    q = levels(kind, n, seed).astype(np.float32)
    if kind == "ties":  # half-way values and their neighbours
        x = q + np.float32(0.5)
        r = np.random.Generator(np.random.PCG64(seed + 1))
        s = r.integers(0, 3, n)
        x = np.where(s == 0, x, np.where(s == 1, np.nextafter(x, np.float32(1e9)), q)).astype(np.float32)
    else:
        x = q
    t = torch.from_numpy(x)
    return t.to(torch.bfloat16) if dtype == "bf16" else t


def host(t):
    return workloads.bf16_bits(t) if t.dtype == torch.bfloat16 else t.numpy()


def shifted(t, off):
    """The same values at an address `off` elements past a 16-byte boundary."""
    b = torch.zeros(t.numel() + 16, dtype=t.dtype, device="cuda")
    b[off:off + t.numel()] = t.cuda()
    return b[off:off + t.numel()]


@pytest.mark.parametrize("block", BLOCKS)
@pytest.mark.parametrize("kind", KINDS)
def test_streams_and_values(zc, block, kind):
    lg = block.bit_length() - 1
    for i, n in enumerate(SIZES):
        for dtype in ("f32", "bf16"):
            x = values(kind, n, 100 * i + block, dtype)
            off = i % 4
            xd = shifted(x, off)
            ref = oracle.compress(host(x), EB, lg)
            out, ob = zc.compress(xd, EB, block)
            assert zc.stream_bytes(out, ob) == ref, (n, dtype)
            y = shifted(torch.zeros(n, dtype=x.dtype), (i + 1) % 4)
            zc.decompress(out, n, out=y)
            want = oracle.decompress(ref, n, out_dtype=oracle.BF16 if dtype == "bf16" else oracle.F32)
            np.testing.assert_array_equal(host(y.cpu()), want)


@pytest.mark.parametrize("block", BLOCKS)
@pytest.mark.parametrize("kind", ["d8", "d16", "wide", "mixed", "offset"])
def test_heads_apart(zc, block, kind):
    lg = block.bit_length() - 1
    for i, n in enumerate(SIZES):
        x = values(kind, n, 7 * i + block, "f32")
        ref = oracle.compress_heads(x.numpy(), EB, lg)
        out, ob = zc.compress(shifted(x, i % 4), EB, block, heads=True)
        assert zc.stream_bytes(out, ob) == ref, n
        y = zc.decompress(out, n)
        np.testing.assert_array_equal(y.cpu().numpy(), oracle.decompress(ref, n))


@pytest.mark.parametrize("block", BLOCKS)
@pytest.mark.parametrize("kind", ["d8", "d16", "wide", "edge8", "ties"])
def test_fused_step(zc, block, kind):
    lg = block.bit_length() - 1
    for i, n in enumerate(SIZES):
        x = values(kind, n, 11 * i + block, "f32")
        loc = values(kind, n, 13 * i + block, "f32")
        cin = oracle.compress(x.numpy(), EB, lg)
        buf = torch.zeros((len(cin) + 15) // 16 * 16, dtype=torch.uint8, device="cuda")
        buf[:len(cin)] = torch.from_numpy(np.frombuffer(cin, np.uint8).copy()).cuda()
        s = shifted(torch.zeros(n), (i + 2) % 4)
        out, ob, sm = zc.reduce_step(buf, shifted(loc, i % 4), EB, block, want_sum=True, sum_out=s)
        ref, ref_sum = oracle.reduce_step(cin, loc.numpy(), EB, lg, want_stream=True, want_sum=True)
        assert zc.stream_bytes(out, ob) == ref, n
        np.testing.assert_array_equal(sm.cpu().numpy(), ref_sum)
        only = zc.reduce_step(buf, shifted(loc, i % 4), EB, block, want_stream=False, want_sum=True)[2]
        np.testing.assert_array_equal(only.cpu().numpy(), ref_sum)


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf"), 4194305.0, 1e30])
def test_errors_in_any_row(zc, bad):
    for at in (0, 31, 32, 1023, 1500):
        x = torch.zeros(1600)
        x[at] = bad
        ws = zc.Workspace(1600)
        zc.compress(x.cuda(), EB, 32, ws=ws)
        st, _ = ws.status()
        assert st == (zc.ERR_RANGE if abs(bad) < 2e30 else zc.ERR_NONFINITE), (bad, at)
