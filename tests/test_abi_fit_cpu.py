"""Argument checks of zc_mlp_fit_epoch (CPU only): each call fails before any CUDA
call and never dereferences the placeholder addresses."""

import pytest

FAKE = 1 << 20


@pytest.fixture(scope="module")
def zc():
    from paper_2308_05199_gb300 import build as zbuild
    zbuild.build()
    from paper_2308_05199_gb300 import zc as z
    return z


@pytest.mark.parametrize("N,batch", [(1000, 256), (1000, 64), (5000, 2000), (100, 256)])
def test_fit_epoch_arguments(zc, N, batch):
    need = zc.zc_mlp_scratch_bytes(min(N, batch))
    names = ["d_params", "d_vel", "d_grad", "d_norm", "d_x", "d_t", "d_idx"]

    def fit(N=N, batch=batch, losses=FAKE, scratch=FAKE, sb=need, **null):
        p = [null.get(k, FAKE) for k in names]
        return zc.zc_mlp_fit_epoch(*p, N, batch, 0.1, 0.9, losses, scratch, sb, None)

    for k in names:
        assert fit(**{k: None}) == zc.ERR_ARG, k
    assert fit(losses=None) == zc.ERR_ARG
    assert fit(N=-1) == zc.ERR_ARG
    assert fit(batch=0) == zc.ERR_ARG
    assert fit(N=0, scratch=None, sb=0) == zc.OK  # nothing to do
    assert fit(scratch=None) == zc.ERR_ARG
    assert fit(scratch=FAKE + 2) == zc.ERR_ARG
    assert fit(sb=need - 1) == zc.ERR_ARG
