"""The library's own choice of the row-resident kernel: calls captured into a graph before and after the stream has its
scratch, and a later, larger layer that leaves the captured graphs valid."""
import numpy as np
import pytest
import torch

from paper_2505_03254_b200 import binding
from gpu_util import make_case, oracle_y, to_device

pytestmark = pytest.mark.gpu


def test_capture_before_and_after_the_scratch_exists(oracle):
    m = 148 * 128                                        # one row tile per SM: the row-resident kernel's smallest
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
