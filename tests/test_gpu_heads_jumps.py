"""Heads apart, rows that begin far from the end of the row before (blocks of
several rows): what the rest of such a row holds is still told apart.  Bad
values give the oracle's error, good ones far from 0 its stream."""

import numpy as np
import pytest
import torch

import oracle
from paper_2308_05199_gb300 import workloads

pytestmark = pytest.mark.gpu

EB = 0.5  # 2 eb = 1: levels are the values' nearest integers
N = 3 * 1024 + 40


@pytest.fixture(scope="module")
def zc():
    from paper_2308_05199_gb300 import build as zbuild, zc as z
    zbuild.build()
    return z


def host(t):
    return workloads.bf16_bits(t) if t.dtype == torch.bfloat16 else t.numpy()


@pytest.mark.parametrize("value", [float("nan"), float("inf"), float("-inf"), 1e30, 6e6, 3e6, 40000.0])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("block", [16, 32, 64, 128])
def test_values_behind_a_jump(zc, block, dtype, value):
    for level in (20000.0, float(1 << 21)):
        for rows in ([3], list(range(1, N // 32, 2))):  # one such row, and every other one
            for at in (1, 7, 31):
                x = torch.zeros(N)
                for r in rows:
                    x[32 * r:32 * r + 32] = level
                    x[32 * r + at] = value
                x = x.to(dtype)
                try:
                    want, ref = 0, oracle.compress_heads(host(x), EB, block.bit_length() - 1)
                except oracle.OracleError as e:
                    want = e.status
                ws = zc.Workspace(N)
                out, ob = zc.compress(x.cuda(), EB, block, ws=ws, heads=True)
                assert ws.status()[0] == want, (level, len(rows), at)
                if want == 0:
                    assert zc.stream_bytes(out, ob) == ref
