"""Segments of every length and alignment from the encoder's ring to the
stream: large tiles (several rounds through the group buffer), wide and narrow
deltas (segments of a few bytes to beyond one round), every block size (units
of 2 to 16 bytes), byte for byte against the oracle."""

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture
def zc():
    from paper_2308_05199_gb300 import build as zbuild, zc as z
    zbuild.build()
    yield z
    z.zc_set_tile_chunks(0)


@pytest.mark.parametrize("block", [16, 32, 64, 128])
@pytest.mark.parametrize("chunks", [4, 8, 16])
def test_segments(zc, chunks, block):
    zc.zc_set_tile_chunks(chunks)
    r = np.random.Generator(np.random.PCG64(block + chunks))
    for n in (chunks * 2048 * 3 + 1, chunks * 2048 + 1023):
        # per block of 128: zero, narrow or the widest levels, so that segment
        # ends fall on any unit
        kind = np.repeat(r.choice([0, 1, 2, 3], n // 128 + 1, p=[.2, .3, .3, .2]), 128)[:n]
        q = np.where(kind == 0, 0, np.where(kind == 1, r.integers(-3, 4, n),
                     np.where(kind == 2, r.integers(-(1 << 20), 1 << 20, n), r.integers(-500, 500, n))))
        for x in (q.astype(np.float32), np.where(kind == 0, 0, r.integers(-(1 << 21), 1 << 21, n)).astype(np.float32)):
            out, ob = zc.compress(torch.from_numpy(x).cuda(), 0.5, block)
            assert zc.stream_bytes(out, ob) == oracle.compress(x, 0.5, block.bit_length() - 1), n
