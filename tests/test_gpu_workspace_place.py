"""Workspaces that start on any 16-byte boundary: the staged payloads of many
tiles per encoder CTA, at every unit size and block size, against the oracle."""

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def zc():
    from paper_2308_05199_gb300 import build as zbuild, zc as z
    zbuild.build()
    yield z
    z.zc_set_tile_chunks(0)


def workspace(zc, n, off):
    w = zc.Workspace.__new__(zc.Workspace)
    w.nbytes = zc.zc_workspace_bytes(n, 1)
    base = torch.empty(w.nbytes + 256, dtype=torch.uint8, device="cuda")
    off += -base.data_ptr() % 128
    w.buf = base[off:off + w.nbytes]
    assert zc.zc_workspace_init(w.ptr, w.nbytes, torch.cuda.current_stream().cuda_stream) == 0
    return w


@pytest.mark.parametrize("off", [0, 16, 64, 112])
@pytest.mark.parametrize("chunks", [4, 8, 16])
def test_any_16_byte_boundary(zc, chunks, off):
    n = 456 * 2048 * chunks * 3 // 2 + 77  # more tiles than CTAs: ring slots are used again
    r = np.random.default_rng(chunks + off)
    x = (r.standard_normal(n) * 0.05).astype(np.float32)
    xd = torch.from_numpy(x).cuda()
    zc.zc_set_tile_chunks(chunks)
    ws = workspace(zc, n, off)
    for block in (16, 32, 64, 128):
        out, ob = zc.compress(xd, 1e-3, block, ws=ws)
        ref = oracle.compress(x, 1e-3, block.bit_length() - 1)
        assert zc.stream_bytes(out, ob) == ref, block
        out2, ob2, _ = zc.reduce_step(out, xd, 1e-3, block, ws=ws)
        ref2 = oracle.reduce_step(ref, x, 1e-3, block.bit_length() - 1, want_stream=True)[0]
        assert zc.stream_bytes(out2, ob2) == ref2, block
        y = zc.decompress(out, n, ws=ws)
        np.testing.assert_array_equal(y.cpu().numpy(), oracle.decompress(ref, n))
    assert ws.status()[0] == 0
