"""The zero padding behind a stream's width bytes: a byte no width can have is a format
error wherever it lies, also beyond the last group of rows (blocks of 128), and a
smaller one makes the widths' sum differ from the header's payload size."""

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

EB = 1e-3


@pytest.fixture(scope="module")
def zc():
    from paper_2308_05199_gb300 import build as zbuild, zc as z
    zbuild.build()
    return z


def stream(n, block, at, value):
    """A stream of n elements with padding byte `at` behind the last width set."""
    x = (np.random.default_rng(n).standard_normal(n) * 0.05).astype(np.float32)
    s = bytearray(oracle.compress(x, EB, block.bit_length() - 1))
    nb = -(-n // block)
    pad = -nb % 16
    if at >= pad:
        return None
    s[32 + nb + at] = value
    return x, torch.frombuffer(s, dtype=torch.uint8).cuda()


@pytest.mark.parametrize("value", [25, 200, 3])
@pytest.mark.parametrize("n", [1024, 3 * 1024, 17 * 1024, 81 * 1024, 300 * 1024 + 5])
@pytest.mark.parametrize("block", [16, 32, 64, 128])
def test_padding_bytes(zc, block, n, value):
    for at in (0, 7, 14):
        made = stream(n, block, at, value)
        if made is None:
            continue
        x, s = made
        ws = zc.Workspace(n)
        zc.decompress(s, n, ws=ws)
        assert ws.status()[0] == zc.ERR_FORMAT, at
        ws.clear()
        zc.reduce_step(s, torch.from_numpy(x).cuda(), EB, block, ws=ws)
        assert ws.status()[0] == zc.ERR_FORMAT, at
        off = torch.tensor([0, s.numel()], dtype=torch.int64, device="cuda")
        d = zc.BatchDecompress(s, off, [torch.zeros(n, device="cuda")])
        d.run()
        assert d.ws.status()[0] == zc.ERR_FORMAT, at


@pytest.mark.parametrize("n", [9, 500, 17 * 1024, 4 * 16384 - 700])
@pytest.mark.parametrize("block", [16, 32, 64, 128])
def test_small_items_of_a_batch(zc, block, n):
    """Widths in the padding of a batch's small items are let through where the planes
    they stand for would lie inside the item's room, and change no value."""
    made = stream(n, block, 0, 2)
    if made is None:
        pytest.skip("no padding at this size")
    x, s = made
    room = torch.zeros(s.numel() + 1024, dtype=torch.uint8, device="cuda")
    room[:s.numel()] = s
    off = torch.tensor([0, room.numel()], dtype=torch.int64, device="cuda")
    y = torch.zeros(n, device="cuda")
    d = zc.BatchDecompress(room, off, [y])
    d.run()
    assert d.ws.status()[0] == 0
    good = oracle.decompress(oracle.compress(x, EB, block.bit_length() - 1), n)
    np.testing.assert_array_equal(y.cpu().numpy(), good)
    ws = zc.Workspace(n)
    zc.decompress(room, n, ws=ws)
    assert ws.status()[0] == zc.ERR_FORMAT
