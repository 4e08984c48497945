"""The library's own choice of the row-resident kernel: calls captured into a graph before and after the stream has its
scratch, and a later, larger layer that leaves the captured graphs valid."""
import numpy as np
import pytest
import torch

from paper_2505_03254_b200 import binding
from gpu_util import make_case, oracle_y, to_device

pytestmark = pytest.mark.gpu


def test_capture_before_and_after_the_scratch_exists(oracle):
    m = 148 * 128                                        # well above the 40 rows per SM from which it is the kernel's
    x, lay = make_case(3, m, 640, 256)
    xd, wp, consts = to_device(x, lay)
    rq = binding.make_requant(*consts)
    want = torch.from_numpy(oracle_y(oracle, x, lay)).cuda()
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    graphs = []
    y = torch.empty((m, 256), dtype=torch.int8, device="cuda")
    for _ in range(2):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            binding.pw_conv_i8(xd, wp, 256, rq, y=y)
        graphs.append(g)
        with torch.cuda.stream(side):                    # now the stream has scratch
            binding.pw_conv_i8(xd, wp, 256, rq)
        side.synchronize()
    big, blay = make_case(4, m, 1024, 1280)              # needs a larger one
    bx, bwp, bconsts = to_device(big, blay)
    with torch.cuda.stream(side):
        by = binding.pw_conv_i8(bx, bwp, 1280, binding.make_requant(*bconsts))
    side.synchronize()
    for g in graphs:
        y.fill_(-77)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, want)
    rows = np.r_[0:256, m - 256:m]
    assert np.array_equal(by.cpu().numpy()[rows], oracle.conv_mul(big.numpy()[rows], blay["w"].numpy(), blay["bias"].numpy(),
                                                                  blay["mult"].numpy(), blay["shift"].numpy(), 0, 127))
    assert binding.last_device_status() == binding.PROM_OK


@pytest.mark.parametrize("cout", [256, 720, 960])
@pytest.mark.parametrize("m", [148 * 128 - 1, 148 * 128, 148 * 128 + 1, 25088])
def test_around_the_choice(oracle, m, cout):
    x, lay = make_case(m + cout, m, 640, cout)
    xd, wp, consts = to_device(x, lay)
    y = binding.pw_conv_i8(xd, wp, cout, binding.make_requant(*consts))
    torch.cuda.synchronize()
    rows = np.r_[0:300, m // 2:m // 2 + 300, m - 300:m]
    want = oracle.conv_mul(x.numpy()[rows], lay["w"].numpy(), lay["bias"].numpy(), lay["mult"].numpy(), lay["shift"].numpy(), 0, 127)
    assert np.array_equal(y.cpu().numpy()[rows], want)


def _rows(per_sm):
    return per_sm * torch.cuda.get_device_properties(0).multi_processor_count


def _launches(m, cin, cout, lo, hi):
    """How many kernels a plain call launches (1: weight-resident, 2: operands and row-resident kernel), its result
    checked against the plain kernel."""
    x, lay = make_case(m + cin + cout, m, cin, cout)
    xd, wp, consts = to_device(x, lay)
    rq = binding.make_requant(*consts, lo, hi)
    want = binding.pw_conv_i8(xd, wp, cout, rq, variant="naive")
    before = binding.launch_count()
    y = binding.pw_conv_i8(xd, wp, cout, rq)
    n = binding.launch_count() - before
    assert torch.equal(y, want)
    return n


@pytest.mark.parametrize("lo", [0, -128])
@pytest.mark.parametrize("per_sm,cin,cout", [(80, 320, 256), (80, 960, 64), (40, 512, 240), (40, 576, 160), (20, 576, 320)])
def test_rules_of_plain_calls(per_sm, cin, cout, lo):
    m = _rows(per_sm)
    assert _launches(m, cin, cout, lo, 127) == 2
    assert _launches(m - 1, cin, cout, lo, 127) == 1
    assert _launches(m, cin - 16, cout, lo, 127) == 1
    if cout > 64:                                        # (960 inputs: any width from 64 on)
        assert _launches(m, cin, cout - 16, lo, 127) == 1
    assert _launches(m, cin, cout, lo, 126) == 1         # another clamp


@pytest.mark.parametrize("per_sm,cin,cout", [(80, 320, 512), (80, 576, 240), (80, 960, 160), (40, 960, 320), (20, 576, 960)])
def test_rules_of_prepared_calls(per_sm, cin, cout):
    def kernel(m, k, n):
        sizes = []
        for mode in (0, 1, 2):
            binding.debug_tc_wide(mode)
            sizes.append(binding.lib().prom_pw_prepared_bytes(m, k, n))
        binding.debug_tc_wide(0)
        assert sizes[1] != sizes[2]
        return "row-resident" if sizes[0] == sizes[2] else "weight-resident"
    m = _rows(per_sm)
    assert kernel(m, cin, cout) == "row-resident"
    assert kernel(m - 1, cin, cout) == "weight-resident"
    assert kernel(m, cin - 16, cout) == "weight-resident"
    assert kernel(m, cin, cout - 16) == "weight-resident"
