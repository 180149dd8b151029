"""Kernels that start while the one before them still runs read what it wrote:
selections that change every message's block size, each followed at once by the
grouped batch it is for, all launched without a wait in between."""

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

M, EB, ROUNDS = 300, 1e-3, 12


@pytest.fixture(scope="module")
def zc():
    from paper_2308_05199_gb300 import build as zbuild, zc as z
    zbuild.build()
    return z


def test_selections_back_to_back(zc):
    r = np.random.default_rng(5)
    xs = [(r.standard_normal(n) * 0.01).astype(np.float32) for n in r.integers(100, 40000, M)]
    b = zc.BatchCompress([torch.from_numpy(x).cuda() for x in xs], [32] * M, [EB] * M, grouped=True)
    cfg = zc.ZcSelectCfg()
    cfg.link_gbs, cfg.raw_ns_per_byte, cfg.judge_log2 = 12.5, 0.001, 1.0
    for k in range(4):
        cfg.ns_per_byte[k] = 0.001
    # selection s: message i stored raw, or at the block size whose predicted bits are lowest
    kinds = [[(i * i + 3 * i * s + s) % 5 for i in range(M)] for s in range(5)]
    preds, feats = [], []
    for kind in kinds:
        y = np.full((M, 4), 3.0, np.float32)
        for i, k in enumerate(kind):
            y[i] = 6.0 if k == 4 else y[i]
            if k < 4:
                y[i, k] = 0.0
        f = np.zeros((M, zc.N_STATS), np.float32)
        f[:, :4] = 2.0 ** y
        preds.append(torch.from_numpy(y).cuda())
        feats.append(torch.from_numpy(f).cuda())
    s = torch.cuda.current_stream().cuda_stream
    got = [(torch.zeros_like(b.packed), torch.zeros_like(b.msg_off)) for _ in range(ROUNDS)]
    torch.cuda.synchronize()
    for k in range(ROUNDS):
        j = k % 5
        assert zc.zc_batch_select(b.plan, feats[j].data_ptr(), preds[j].data_ptr(), cfg, None, None, s) == 0
        b.run()
        got[k][0].copy_(b.packed)
        got[k][1].copy_(b.msg_off)
    assert b.ws.status()[0] == 0
    want = [[oracle.compress_raw(x) if k == 4 else oracle.compress(x, EB, 4 + k)
             for x, k in zip(xs, kind)] for kind in kinds]
    for k in range(ROUNDS):
        packed, off = got[k][0].cpu().numpy(), got[k][1].cpu().numpy()
        for i, w in enumerate(want[k % 5]):
            assert packed[off[i]:off[i] + len(w)].tobytes() == w, (k, i)
