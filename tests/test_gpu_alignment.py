"""Inputs and outputs at every element offset from a 16-byte boundary, of sizes
around a group of 1024 elements and beyond: range (relative bound), scatter
pack of abutting, separated and overlapping segments, and decompression, byte
for byte against the oracle."""

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


def data(n, dtype, seed):
    r = np.random.Generator(np.random.PCG64(seed))
    x = torch.from_numpy(np.cumsum(r.normal(0, 1, n)).astype(np.float32))
    return x.to(torch.bfloat16) if dtype == "bf16" else x


def host(t):
    return workloads.bf16_bits(t) if t.dtype == torch.bfloat16 else t.numpy()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("block", [16, 32, 64, 128])
def test_offsets(zc, block, dtype):
    for off in range(9):
        for n in (3, 1023, 1024, 1025, 2048, 9000 + off):
            x = data(n, dtype, n + off)
            # the extremes at the ends, so that a missed element changes the bound
            x[0], x[n - 1] = -400.0, 400.0
            buf = torch.full((n + 32,), 1e6, dtype=x.dtype, device="cuda")
            buf[off:off + n] = x.cuda()
            out, ob = zc.compress(buf[off:off + n], 1e-3, block, mode=zc.EB_REL)
            ref = oracle.compress(host(x), 0.8, block.bit_length() - 1)
            assert zc.stream_bytes(out, ob) == ref, (off, n)
            y = torch.full_like(buf, 7.0)
            zc.decompress(out, n, out=y[off:off + n])
            want = oracle.decompress(ref, n, out_dtype=oracle.BF16 if dtype == "bf16" else oracle.F32)
            np.testing.assert_array_equal(host(y[off:off + n].cpu()), want)
            assert bool((y[:off] == 7.0).all()) and bool((y[off + n:] == 7.0).all())


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("layout", ["abutting", "gaps", "overlapping", "empty"])
def test_scatter_segments(zc, layout, dtype):
    n = 41007
    x = data(n, dtype, 5)
    x[n // 2] = 900.0
    counts = {"abutting": [1025, 3, 20000, n - 21028], "gaps": [1000, 7001, 12003],
              "overlapping": [9000, 9001, 30000], "empty": [0, 5000, 0, 20003, 0]}[layout]
    displs = {"abutting": [0, 1025, 1028, 21028], "gaps": [1, 3000, 20001],
              "overlapping": [0, 4501, 1111], "empty": [0, 0, 5000, 5000, 25003]}[layout]
    parts = [x[d:d + c] for c, d in zip(counts, displs)]
    f = torch.cat([p.float() for p in parts])
    eb = float(np.float32(1e-3 * (float(f.max()) - float(f.min()))))
    out, off = zc.scatter_pack(x.cuda(), counts, displs, 1e-3, 32, mode=zc.EB_REL)[:2]
    o = off.cpu().numpy()
    raw = out.cpu().numpy().tobytes()
    for k, p in enumerate(parts):
        ref = oracle.compress(host(p), eb, 5)
        assert raw[o[k]:o[k + 1]][:len(ref)] == ref, k
