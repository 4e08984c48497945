"""The dynamic layer's codes on enough values to meet products next to a rounding tie: the second pass, which
works on pairs of floats, against the definition's single binary32 operations taken by torch on the
accumulators of the plain kernel."""
import pytest
import torch

from paper_2505_03254_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,rows,cin,cout", [(32, 12544, 16, 96), (20, 3136, 64, 256), (64, 784, 144, 40)])
def test_every_operation_rounds_once(batch, rows, cin, cout):
    g = torch.Generator(device="cuda").manual_seed(cin + cout)
    x = torch.randint(-127, 128, (batch * rows, cin), generator=g, device="cuda", dtype=torch.int8)
    wp = binding.pack_ternary(torch.randint(-1, 2, (cout, cin), generator=g, device="cuda", dtype=torch.int8))
    alpha = torch.rand((cout,), generator=g, device="cuda") * 0.2 + 0.01
    gamma = torch.rand((batch,), generator=g, device="cuda") * 7.0 + 0.5
    q, gy, sy = binding.pw_conv_i8_dyn(x, batch, wp, cout, alpha, gamma)
    acc = binding.pw_conv_i8_acc32(x, wp, cout).float()              # exact: below 2^24
    y = (acc * alpha).view(batch, -1) * (gamma / torch.full_like(gamma, 127.0))[:, None]      # each a kernel of its own: nothing is fused
    want_g = y.abs().amax(1)
    want_s = torch.full_like(want_g, 127.0) / want_g                # (torch takes a scalar quotient through a reciprocal)
    assert torch.equal(gy, want_g) and torch.equal(sy, want_s)
    want = torch.round(y * want_s[:, None]).clamp_(-128, 127).to(torch.int8)
    assert torch.equal(q.view(batch, -1), want), int((q.view(batch, -1) != want).sum())
