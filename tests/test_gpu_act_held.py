"""The activation quantiser's clusters whose CTAs keep the first chunks of a slice in registers (slices that fill an SM,
several rounds of samples): codes, gamma and scale bit for bit against the oracle at the edges of the chunks."""
import numpy as np
import pytest
import torch

from paper_2505_03254_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,per", [
    (76, 8 * 29600),           # four chunks, the last of them short
    (70, 8 * 32768),           # four whole chunks
    (70, 8 * 32768 + 16),      # a fifth chunk of a few floats
    (47, 8 * 50176),           # seven chunks
    (42, 8 * 55808 - 112),     # as much as shared memory holds, a ragged last CTA
])
def test_held_chunks(oracle, batch, per):
    assert batch * per * 4 > 64 << 20                  # beyond one group of the grouped route
    rng = np.random.default_rng(per)
    x = rng.standard_normal((batch, per), dtype=np.float32)
    x *= np.exp2(rng.integers(-20, 20, size=(batch, 1))).astype(np.float32)
    x[batch // 3] = 0.0
    x[1, 5] = np.nan                                    # has no part in the maximum
    x[2, per - 1] = np.float32(3e5)
    want_q, want_g, want_s = oracle.quantize_act_absmax(x)
    xd = torch.from_numpy(x).cuda()
    out = (torch.full((batch, per), 77, dtype=torch.int8, device="cuda"), torch.full((batch,), -1.0, device="cuda"),
           torch.full((batch,), -1.0, device="cuda"))
    for _ in range(2):                                  # a second call overlaps the end of the first
        q, g, s = binding.quantize_act_absmax(xd, out=out)
    torch.cuda.synchronize()
    assert binding.last_device_status() == binding.PROM_OK
    assert np.array_equal(g.cpu().numpy().view(np.uint32), want_g.view(np.uint32))
    assert np.array_equal(s.cpu().numpy().view(np.uint32), want_s.view(np.uint32))
    real = ~np.isnan(x)
    assert np.array_equal(q.cpu().numpy()[real], want_q[real])
