"""Arguments that the binding refuses on the host, before anything is launched."""
import pytest
import torch

from paper_2505_03254_b200 import binding

pytestmark = pytest.mark.gpu

M, CIN, COUT = 256, 64, 96


@pytest.fixture(scope="module")
def layer():
    rq = binding.make_requant(torch.zeros(COUT, dtype=torch.int32, device="cuda"),
                              torch.full((COUT,), 1 << 30, dtype=torch.int32, device="cuda"),
                              torch.full((COUT,), 4, dtype=torch.int8, device="cuda"))
    wp = binding.pack_ternary(torch.ones((COUT, CIN), dtype=torch.int8, device="cuda"))
    return torch.zeros((M, CIN), dtype=torch.int8, device="cuda"), wp, rq


def _refused(call, error, what):
    before = binding.launch_count()
    with pytest.raises(error, match=what):
        call()
    assert binding.launch_count() == before


def test_prepared_operands_that_are_not_a_device_buffer(layer):
    x, wp, rq = layer
    good = binding.pw_prepare(M, CIN, wp, COUT, rq)
    for bad in (good.cpu(), good.view(torch.int8), good[::2]):
        _refused(lambda: binding.pw_conv_i8_prepared(x, COUT, bad), ValueError, "prepared")
    binding.pw_conv_i8_prepared(x, COUT, good)
    assert binding.last_device_status() == binding.PROM_OK
