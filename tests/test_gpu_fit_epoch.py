"""A training epoch in one call against the oracle's steps in FP64, and against
the steps launched one by one, bit for bit: minibatches smaller than a tile of
64 rows, exactly one, several, several turns of four tiles, ragged last ones,
and above the size up to which one cluster trains."""

import numpy as np
import pytest
import torch

from oracle import selector as OS

pytestmark = pytest.mark.gpu

LR, MOMENTUM = 0.02, 0.9


@pytest.fixture(scope="module")
def zc():
    from paper_2308_05199_gb300 import build as zbuild, zc as z
    zbuild.build()
    return z


@pytest.mark.parametrize("N,batch", [(1, 1), (5, 64), (300, 64), (1000, 256), (523, 257), (700, 600),
                                     (2047, 2047), (1000, 1000), (900, 65), (2500, 1024), (2500, 1025)])
def test_epoch(zc, N, batch):
    r = np.random.default_rng(N + batch)
    p0 = (OS.init_params(N) + r.normal(0, 0.05, OS.N_PARAMS)).astype(np.float32)
    v0 = r.normal(0, 1e-3, OS.N_PARAMS).astype(np.float32)
    norm = np.concatenate([r.normal(0, 1, 16), r.uniform(0.5, 2, 16)]).astype(np.float32)
    X = r.normal(0, 1, (N, 16)).astype(np.float32)
    T = r.normal(0, 1, (N, 4)).astype(np.float32)
    idx = r.permutation(N).astype(np.int32)
    d = {k: torch.from_numpy(a.copy()).cuda() for k, a in
         dict(p=p0, v=v0, norm=norm, X=X, T=T, idx=idx).items()}
    g = torch.zeros(OS.N_PARAMS, device="cuda")
    steps = (N + batch - 1) // batch
    losses = torch.full((steps + 1,), -1.0, device="cuda")
    scratch = torch.empty(zc.zc_mlp_scratch_bytes(batch) // 4, device="cuda")
    st = zc.zc_mlp_fit_epoch(d["p"].data_ptr(), d["v"].data_ptr(), g.data_ptr(), d["norm"].data_ptr(),
                             d["X"].data_ptr(), d["T"].data_ptr(), d["idx"].data_ptr(), N, batch, LR,
                             MOMENTUM, losses.data_ptr(), scratch.data_ptr(), scratch.numel() * 4,
                             torch.cuda.current_stream().cuda_stream)
    assert st == 0
    # the same steps, one by one
    stream = torch.cuda.current_stream().cuda_stream
    q, w = torch.from_numpy(p0).cuda(), torch.from_numpy(v0).cuda()
    gc, lc = torch.zeros_like(g), torch.zeros(steps, device="cuda")
    for k in range(steps):
        B = min(batch, N - k * batch)
        assert zc.zc_mlp_grad(q.data_ptr(), d["norm"].data_ptr(), d["X"].data_ptr(), d["T"].data_ptr(),
                              d["idx"].data_ptr() + 4 * k * batch, B, gc.data_ptr(), lc.data_ptr() + 4 * k,
                              scratch.data_ptr(), scratch.numel() * 4, stream) == 0
        assert zc.zc_mlp_sgd(q.data_ptr(), w.data_ptr(), gc.data_ptr(), LR, MOMENTUM, stream) == 0
    assert torch.equal(d["p"], q) and torch.equal(d["v"], w)
    assert torch.equal(g, gc) and torch.equal(losses[:steps], lc)
    p, v = p0.astype(np.float64), v0.astype(np.float64)
    ref_loss, gmax = [], 0.0
    for k in range(steps):
        i = idx[k * batch:(k + 1) * batch]
        loss, gr = OS.loss_grad(p, norm.astype(np.float64), X[i].astype(np.float64), T[i].astype(np.float64))
        v = MOMENTUM * v + gr
        p = p - LR * v
        ref_loss.append(loss)
        gmax = max(gmax, float(np.max(np.abs(gr))))
    # every step's gradient within 1e-4 of the largest entry, as for one
    # gradient; velocity and parameters add them up
    tol = 1e-4 * gmax * steps
    assert np.max(np.abs(g.cpu().numpy() - gr)) <= tol
    assert np.max(np.abs(d["v"].cpu().numpy() - v)) <= tol
    assert np.max(np.abs(d["p"].cpu().numpy() - p)) <= LR * tol * steps + 1e-6
    np.testing.assert_allclose(losses[:steps].cpu().numpy(), ref_loss, rtol=1e-4)
    assert losses[steps].item() == -1.0
