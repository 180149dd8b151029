"""Streams whose unit offsets are found without a width scan (small single
streams, launches of few tiles) on both sides of every limit: values against
the oracle, bad streams and workspaces reported as with the scan."""

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

TILE = 16384


@pytest.fixture(scope="module")
def zc():
    from paper_2308_05199_gb300 import build as zbuild, zc as z
    zbuild.build()
    z.zc_set_tile_chunks(0)
    return z


def signal(n, seed):
    r = np.random.Generator(np.random.PCG64(seed))
    # widths that differ from block to block
    s = np.repeat(r.choice([0, 1, 9, 300, 40000], n // 100 + 1), 100)[:n]
    return (r.integers(-1000, 1000, n) * s / 1000.0).astype(np.float32)


@pytest.mark.parametrize("block", [16, 32, 64, 128])
@pytest.mark.parametrize("n", [1, TILE - 1, TILE + 1, 9 * TILE + 777, 256 * TILE, 256 * TILE + 1])
def test_single_stream(zc, n, block):
    x = signal(n, n + block)
    out, ob = zc.compress(torch.from_numpy(x).cuda(), 0.5, block)
    ref = oracle.compress(x, 0.5, block.bit_length() - 1)
    assert zc.stream_bytes(out, ob) == ref
    y = zc.decompress(out, n)
    np.testing.assert_array_equal(y.cpu().numpy(), oracle.decompress(ref, n))


@pytest.mark.parametrize("block,n", [(16, 1 << 20), (16, (1 << 20) + 1), (32, 100003), (128, (1 << 20) + 5),
                                     (128, 8192 * 1024), (128, 8192 * 1024 + 1)])
def test_fused_step(zc, block, n):
    lg = block.bit_length() - 1
    a, b = signal(n, 3), signal(n, 4)
    cin = oracle.compress(a, 0.5, lg)
    buf = torch.from_numpy(np.frombuffer(cin, np.uint8).copy()).cuda()
    out, ob, sm = zc.reduce_step(buf, torch.from_numpy(b).cuda(), 0.5, block, want_sum=True)
    ref, ref_sum = oracle.reduce_step(cin, b, 0.5, lg, want_stream=True, want_sum=True)
    assert zc.stream_bytes(out, ob) == ref
    np.testing.assert_array_equal(sm.cpu().numpy(), ref_sum)


@pytest.mark.parametrize("sizes", [[5 * TILE + 1, 3, TILE * 128, TILE * 129], [TILE * 100] * 10 + [TILE * 24],
                                   [TILE * 100] * 10 + [TILE * 24 + 1]])
def test_batch(zc, sizes):
    xs = [signal(n, i) for i, n in enumerate(sizes)]
    dev = [torch.from_numpy(x).cuda() for x in xs]
    comp = zc.BatchCompress(dev, [32] * len(xs), [0.5] * len(xs))
    packed, off = comp.run()
    outs = [torch.empty_like(d) for d in dev]
    zc.BatchDecompress(packed, off, outs, ws=comp.ws).run()
    for x, y in zip(xs, outs):
        np.testing.assert_array_equal(y.cpu().numpy(), oracle.decompress(oracle.compress(x, 0.5, 5), x.size))
    assert comp.ws.status()[0] == 0


def test_bad_streams_and_workspaces(zc):
    n = 3 * TILE + 100
    x = torch.from_numpy(signal(n, 1)).cuda()
    good, ob = zc.compress(x, 0.5, 32)
    good = good[:int(ob)].clone()
    for at, value in ((24, 0xff), (32 + 40, 25), (32 + 40, 255)):  # payload size; a width beyond the format's
        bad = good.clone()
        bad[at] = value
        for call in (lambda ws: zc.decompress(bad, n, ws=ws),
                     lambda ws: zc.reduce_step(bad, x, 0.5, 32, want_sum=True, ws=ws)):
            ws = zc.Workspace(n, 1)
            call(ws)
            assert ws.status()[0] == zc.ERR_FORMAT, (at, value)
    ws = zc.Workspace(n, 1)
    ws.buf.zero_()
    zc.decompress(good, n, ws=ws)
    assert ws.status()[0] == zc.ERR_WORKSPACE
