"""zc_mlp_fit_epoch without proper scratch is an argument error on every route, and
nothing is trained."""

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def zc():
    from paper_2308_05199_gb300 import build as zbuild, zc as z
    zbuild.build()
    return z


@pytest.mark.parametrize("N,batch", [(300, 64), (100, 256), (2500, 2000)])
def test_scratch_is_checked(zc, N, batch):
    f = lambda *s: torch.ones(*s, device="cuda")  # noqa: E731
    p, v, g, norm, X, T = f(zc.MLP_PARAMS), f(zc.MLP_PARAMS), f(zc.MLP_PARAMS), f(32), f(N, 16), f(N, 4)
    idx, losses = torch.arange(N, dtype=torch.int32, device="cuda"), f(N)
    need = zc.zc_mlp_scratch_bytes(min(N, batch))
    scratch = f(need // 4 + 1)
    s = torch.cuda.current_stream().cuda_stream

    def fit(ptr, nbytes):
        return zc.zc_mlp_fit_epoch(p.data_ptr(), v.data_ptr(), g.data_ptr(), norm.data_ptr(), X.data_ptr(),
                                   T.data_ptr(), idx.data_ptr(), N, batch, 0.01, 0.9, losses.data_ptr(),
                                   ptr, nbytes, s)

    assert fit(None, need) == zc.ERR_ARG
    assert fit(scratch.data_ptr(), need - 1) == zc.ERR_ARG
    assert fit(scratch.data_ptr() + 2, need) == zc.ERR_ARG
    assert bool((p == 1).all()) and bool((losses == 1).all())
    assert fit(scratch.data_ptr(), need) == zc.OK
    assert not bool((p == 1).all())
