"""The bound of a relative scatter pack of many segments with gaps between them: the
extremes lie at the first and last elements of segments that start anywhere, and
values beyond them in the gaps do not count."""

import numpy as np
import pytest
import torch

import oracle
from paper_2308_05199_gb300 import workloads

pytestmark = pytest.mark.gpu

REL = 1e-2


@pytest.fixture(scope="module")
def zc():
    from paper_2308_05199_gb300 import build as zbuild, zc as z
    zbuild.build()
    return z


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("P,lo,hi", [(2, 1, 9), (17, 0, 30), (49, 1, 200), (400, 1, 40), (9, 5000, 90000)])
def test_extremes_at_the_ends(zc, P, lo, hi, dtype):
    r = np.random.default_rng(P)
    counts = [int(c) for c in r.integers(lo, hi, P)]
    gaps = r.integers(1, 12, P)
    displs = [int(d) for d in np.cumsum(gaps) + np.concatenate([[0], np.cumsum(counts)[:-1]])]
    n = displs[-1] + counts[-1] + 5
    full = [p for p in range(P) if counts[p] >= 2]
    x0 = r.uniform(-1.0, 1.0, n).astype(np.float32)
    inside = np.zeros(n, bool)
    for c, d in zip(counts, displs):
        inside[d:d + c] = True
    x0[~inside] = 1e6
    for p in r.choice(full, min(4, len(full)), replace=False):
        x = x0.copy()
        x[displs[p]], x[displs[p] + counts[p] - 1] = 3.0, -5.0
        t = torch.from_numpy(x).to(dtype)
        h = workloads.bf16_bits(t) if dtype == torch.bfloat16 else x
        out, off = zc.scatter_pack(t.cuda(), counts, displs, REL, 32, mode=zc.EB_REL)[:2]
        eb = oracle.eb_from_rel(REL, -5.0, 3.0)
        o, b = off.cpu().numpy(), out.cpu().numpy()
        for k in range(P):
            ref = oracle.compress(np.ascontiguousarray(h[displs[k]:displs[k] + counts[k]]), eb, 5)
            assert b[o[k]:o[k + 1]].tobytes() == ref, (p, k)
