"""Bounds so large that q 2eb of the largest values overflows FP32: streams with
and without values at exact ties beside them, against the oracle."""

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

FMAX = np.finfo(np.float32).max


@pytest.fixture(scope="module")
def zc():
    from paper_2308_05199_gb300 import build as zbuild, zc as z
    zbuild.build()
    return z


# bounds on both sides of 2 eb = 2^107, up to the largest the codec takes
@pytest.mark.parametrize("eb", [0.75 * 2.0 ** 106, 2.0 ** 107, 1.3 * 2.0 ** 112, 0.75 * 2.0 ** 126, 0.9 * 2.0 ** 126])
@pytest.mark.parametrize("heads", [False, True])
@pytest.mark.parametrize("block", [16, 32, 64, 128])
def test_largest_values(zc, block, heads, eb):
    lg = block.bit_length() - 1
    r = np.random.default_rng(block)
    q = np.floor(min(float(FMAX) / (2 * eb) + 0.5, 60.0))
    for n in (5, 1024, 3000):
        x = (r.integers(-q, q + 1, n) * (2 * eb)).clip(-float(FMAX), float(FMAX)).astype(np.float32)
        x[r.random(n) < 0.1] = FMAX if float(FMAX) / (2 * eb) < 2 ** 21 else 0
        x[r.random(n) < 0.1] = np.float32(eb)  # half-way between levels 0 and 1
        x[0] = -np.float32(eb)
        ref = (oracle.compress_heads if heads else oracle.compress)(x, eb, lg)
        ws = zc.Workspace(n)
        out, ob = zc.compress(torch.from_numpy(x).cuda(), eb, block, ws=ws, heads=heads)
        assert ws.status()[0] == 0
        assert zc.stream_bytes(out, ob) == ref, n
        y = zc.decompress(out, n, ws=ws)
        np.testing.assert_array_equal(y.cpu().numpy(), oracle.decompress(ref, n))
