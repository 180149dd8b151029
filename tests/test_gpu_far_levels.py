"""Streams whose levels lie beyond 2^22, which no encoder here writes but the format
can hold (wide deltas that add up, heads of 24 bits): decoded as the oracle does."""

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

EB = 0.5


@pytest.fixture(scope="module")
def zc():
    from paper_2308_05199_gb300 import build as zbuild, zc as z
    zbuild.build()
    return z


def shifted(s, n, block, heads, r):
    """The stream with some blocks' heads moved far out (heads apart), or with the sign
    planes of some blocks cleared: all their deltas then add up."""
    s, nb, head = bytearray(s), -(-n // block), 32 + (-(-n // block) + 15) // 16 * 16
    if heads:
        for b in r.choice(nb, max(1, nb // 3), replace=False):
            s[head + 3 * b:head + 3 * b + 3] = int(r.integers(-(1 << 23), 1 << 23)).to_bytes(3, "little", signed=True)
        return bytes(s)
    pos = head
    for b in range(nb):
        w = s[32 + b]
        if w and r.random() < 0.5:
            s[pos:pos + block // 8] = bytes(block // 8)
        pos += (w + 1) * (block // 8) if w else 0
    return bytes(s)


@pytest.mark.parametrize("scale", [20, 3000, 100000, 4000000])
@pytest.mark.parametrize("heads", [False, True])
@pytest.mark.parametrize("block", [16, 32, 64, 128])
def test_decoded_as_the_oracle(zc, block, heads, scale):
    r = np.random.default_rng(block + scale)
    for n in (40, 1024, 20000):
        x = r.integers(-scale, scale + 1, n).astype(np.float32)
        lg = block.bit_length() - 1
        s = shifted((oracle.compress_heads if heads else oracle.compress)(x, EB, lg), n, block, heads, r)
        d = torch.frombuffer(bytearray(s), dtype=torch.uint8).cuda()
        ws = zc.Workspace(n)
        y = zc.decompress(d, n, ws=ws)
        assert ws.status()[0] == 0
        np.testing.assert_array_equal(y.cpu().numpy(), oracle.decompress(s, n))
        if not heads:
            local = r.integers(-scale, scale + 1, n).astype(np.float32)
            sm = zc.reduce_step(d, torch.from_numpy(local).cuda(), EB, block, want_stream=False, want_sum=True, ws=ws)[2]
            assert ws.status()[0] == 0
            ref = oracle.reduce_step(s, local, EB, lg, want_stream=False, want_sum=True)[1]
            np.testing.assert_array_equal(sm.cpu().numpy(), ref)
