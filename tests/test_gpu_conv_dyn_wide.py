"""The dynamic layer where one CTA holds more columns than its threads request constants of up front (four per
thread, 1280 in all): the planner takes such plans on a million rows, here they are asked for on a few hundred."""
import pytest
import torch

from paper_2505_03254_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cin,cout,nt", [(16, 1280, 128), (16, 1568, 224), (32, 1760, 160)])
def test_more_columns_than_threads_hold_constants_of(oracle, cin, cout, nt):
    batch, rows = 3, 150
    g = torch.Generator().manual_seed(cout)
    x = torch.randint(-127, 128, (batch * rows, cin), generator=g, dtype=torch.int8)
    w = torch.randint(-1, 2, (cout, cin), generator=g, dtype=torch.int8)
    alpha = torch.rand((cout,), generator=g) * 0.2 + 0.01
    gamma = torch.rand((batch,), generator=g) * 7.0 + 0.5
    want_q, want_g, want_s, _ = oracle.conv_dyn(x.numpy(), w.numpy(), alpha.numpy(), gamma.numpy(), rows)
    binding.debug_tc_plan_shape(batch * rows, cin, cout, nt=nt, groups=1, occ=1)
    try:
        q, gy, sy = binding.pw_conv_i8_dyn(x.cuda(), batch, binding.pack_ternary(w.cuda()), cout, alpha.cuda(), gamma.cuda())
        assert binding.last_device_status() == binding.PROM_OK
    finally:
        binding.debug_tc_plan_shape(batch * rows, cin, cout)
    assert (q.cpu().numpy() == want_q).all() and (gy.cpu().numpy() == want_g).all() and (sy.cpu().numpy() == want_s).all()
