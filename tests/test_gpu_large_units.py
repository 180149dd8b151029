"""Decoder units of 128 rows (launches of 2^26 elements and more), ragged ends
included: single streams against the oracle, a batch against its messages
decoded one by one (64-row units)."""

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
    z.zc_set_tile_chunks(0)
    return z


@pytest.mark.parametrize("block,heads,tail", [(16, False, 0), (32, False, 1), (64, True, 1025), (128, False, 29 * 1024 + 3)])
def test_single_stream(zc, block, heads, tail):
    n = (1 << 26) + tail
    x = workloads.student_t3(n, 1.0, block, device="cuda")
    out, ob = zc.compress(x, 1e-2, block, heads=heads)
    y = zc.decompress(out, n)
    ref = oracle.decompress(zc.stream_bytes(out, ob), n)
    np.testing.assert_array_equal(y.cpu().numpy(), ref)


def test_batch(zc):
    r = np.random.Generator(np.random.PCG64(3))
    sizes = [int(s) for s in r.integers(1_400_000, 2_300_000, 41)] + [1, 32769, 3 * 32768 + 1025, 5 * 32768]
    xs = [workloads.student_t3(n, 1.0, i, device="cuda") for i, n in enumerate(sizes)]
    xs = [x.to(torch.bfloat16) if i % 3 == 0 else x for i, x in enumerate(xs)]
    blocks = [(16, 32, 64, 128, zc.RAW)[i % 5] for i in range(len(xs))]
    assert sum(sizes) >= 1 << 26 and sum(sizes) // len(sizes) >= 1 << 17
    comp = zc.BatchCompress(xs, blocks, [1e-2] * len(xs))
    packed, off = comp.run()
    outs = [torch.zeros_like(x) for x in xs]
    zc.BatchDecompress(packed, off, outs, ws=comp.ws).run()
    assert comp.ws.status()[0] == 0
    o = off.tolist()
    for i, (x, y) in enumerate(zip(xs, outs)):
        one = zc.decompress(packed[o[i]:o[i + 1]].clone(), x.numel(), out=torch.empty_like(x))
        assert torch.equal(y, one), i
