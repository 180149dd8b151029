"""Raw messages of a batch, there and back: every tile size, sizes around a warp's
share and a tile, inputs and outputs off 16- and 4-byte boundaries, between coded
messages, against the oracle."""

import numpy as np
import pytest
import torch

import oracle
from paper_2308_05199_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def zc():
    from paper_2308_05199_gb300 import build as zbuild, zc as z
    zbuild.build()
    return z


def host(t):
    return workloads.bf16_bits(t) if t.dtype == torch.bfloat16 else t.cpu().numpy()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("chunks", [4, 8, 16])
def test_raw_between_coded(zc, chunks, dtype):
    te = 2048 * chunks
    sizes = [1, 7, 8, 1023, te // 8, te // 8 + 1, te - 1, te, te + 1, 3 * te + te // 8 + 13]
    g = torch.Generator(device="cuda")
    g.manual_seed(chunks)
    xs, blocks = [], []
    for i, n in enumerate(sizes):
        for off in (0, 1, 2, 3):
            x = torch.randn(n + 8, generator=g, device="cuda").to(dtype)[off:off + n]
            xs.append(x)
            blocks.append(zc.RAW if (i + off) % 3 else 32)
    b = zc.BatchCompress(xs, blocks, [1e-2] * len(xs), tile_chunks=chunks)
    packed, off = b.run()
    ys = [torch.zeros_like(torch.cat([x, x[:1]]))[1:] for x in xs]
    d = zc.BatchDecompress(packed, off, ys)
    d.run()
    assert b.ws.status()[0] == 0 and d.ws.status()[0] == 0
    p, o = packed.cpu().numpy(), off.cpu().numpy()
    for i, (x, blk) in enumerate(zip(xs, blocks)):
        w = oracle.compress_raw(host(x)) if blk == zc.RAW else oracle.compress(host(x), 1e-2, 5)
        assert p[o[i]:o[i + 1]].tobytes() == w, i
        if blk == zc.RAW:
            np.testing.assert_array_equal(host(ys[i]), host(x))
