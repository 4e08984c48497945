"""The activation quantiser's grouped route (several kernels, codes of one group of samples and then the maxima of
the next) and its choice of cluster sizes: codes, gamma and scale bit for bit against the oracle."""
import numpy as np
import pytest
import torch

from paper_2505_03254_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,per", [
    (1, 4), (3, 1004), (70, 1020), (5, 1028),         # not multiples of 16: pieces of 1024 floats and remainders
    (1, 450560), (2, 500004), (19, 460000),           # beyond eight SMs' shared memory, in one group
    (30, 900004), (3, 16800004),                      # 108 MB: two groups; samples larger than a group
    (200, 94080), (297, 47040), (150, 12288), (37, 100352),   # one and several rounds of clusters
])
def test_routes(oracle, batch, per):
    rng = np.random.default_rng(batch + per)
    x = rng.standard_normal((batch, per), dtype=np.float32)
    x *= np.exp2(rng.integers(-20, 20, size=(batch, 1))).astype(np.float32)
    x[batch // 2] = 0.0                                # an all-zero sample between others
    want_q, want_g, want_s = oracle.quantize_act_absmax(x)
    xd = torch.from_numpy(x).cuda()
    out = (torch.full((batch, per), 77, dtype=torch.int8, device="cuda"), torch.full((batch,), -1.0, device="cuda"),
           torch.full((batch,), -1.0, device="cuda"))
    for _ in range(2):                                 # a second call overlaps the end of the first
        q, g, s = binding.quantize_act_absmax(xd, out=out)
    torch.cuda.synchronize()
    assert np.array_equal(g.cpu().numpy().view(np.uint32), want_g.view(np.uint32))
    assert np.array_equal(s.cpu().numpy().view(np.uint32), want_s.view(np.uint32))
    assert np.array_equal(q.cpu().numpy(), want_q)
    assert binding.last_device_status() == binding.PROM_OK
