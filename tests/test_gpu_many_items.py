"""A fused step over more items than its width scan searches (the scan and the
fused kernel then each take their own item map, in the same workspace array):
every stream and sum against the oracle."""

import numpy as np
import pytest
import torch

import oracle
from paper_2308_05199_gb300 import collectives, zc as z

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("items", [255, 256, 300])
def test_fused_step_of_many_items(items):
    from paper_2308_05199_gb300 import build as zbuild
    zbuild.build()
    z.zc_set_tile_chunks(0)
    r = np.random.Generator(np.random.PCG64(items))
    sizes = [int(n) for n in r.integers(33000, 66000, items)]
    cap = z.zc_max_compressed_bytes(max(sizes), 32)
    xs = [np.cumsum(r.integers(-9, 10, n)).astype(np.float32) % 997 for n in sizes]
    ys = [r.integers(-300, 300, n).astype(np.float32) for n in sizes]
    cins = [oracle.compress(x, 0.5, 5) for x in xs]
    src = torch.zeros((items, cap), dtype=torch.uint8)
    for i, c in enumerate(cins):
        src[i, :len(c)] = torch.from_numpy(np.frombuffer(c, np.uint8).copy())
    src, loc = src.cuda(), [torch.from_numpy(y).cuda() for y in ys]
    dst = torch.zeros_like(src)
    sums = [torch.zeros_like(t) for t in loc]
    nbytes = torch.zeros(items, dtype=torch.int64, device="cuda")
    ws = z.Workspace(sum(sizes), items)
    steps = collectives._Steps(ws, torch.cuda.current_stream())
    steps.reduce([z.ZcReduceItem(src[i].data_ptr(), loc[i].data_ptr(), dst[i].data_ptr(), sums[i].data_ptr(),
                                 nbytes[i].data_ptr(), sizes[i], cap, cap) for i in range(items)],
                 0.5, 32, "step", items)
    for _ in range(3):
        steps.run()
    assert ws.status()[0] == 0
    for i in range(items):
        ref, ref_sum = oracle.reduce_step(cins[i], ys[i], 0.5, 5, want_stream=True, want_sum=True)
        assert dst[i, :int(nbytes[i])].cpu().numpy().tobytes() == ref, i
        np.testing.assert_array_equal(sums[i].cpu().numpy(), ref_sum)
