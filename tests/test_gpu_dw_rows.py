"""The depthwise kernel on TMA and tcgen05 (three tap rows per MMA, output rows streamed through a ring
of accumulators), both strides forced, byte for byte against the oracle."""
import numpy as np
import pytest
import torch

from paper_2505_03254_b200 import binding
from test_gpu_dw import _case, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stride", [1, 2])
@pytest.mark.parametrize("b,h,w,c", [
    (1, 2, 2, 16), (2, 4, 3, 32), (5, 3, 9, 48), (17, 8, 8, 64), (3, 15, 16, 80), (2, 64, 17, 96), (40, 7, 7, 960),
    (150, 33, 9, 64), (9, 5, 130, 144),
])
def test_rows_streamed_through_the_accumulators(oracle, stride, b, h, w, c):
    """One and two slices of a channel block, a last slice of 16 channels, groups that end inside the row
    and tiles that end inside the batch, shares of a few rows up to several tiles per CTA (150 images of
    33 rows), odd and even sizes; mixed shifts and a bias beyond the digits."""
    x, wt, bias, mult, shift = _case(43, b, h, w, c)
    try:
        binding.debug_dw_variant(2)
        for lo, hi in ((0, 127), (-128, 127)):
            _run(oracle, x, wt, bias, mult, shift, stride, lo, hi)
        shift[:] = np.arange(c) % 9 + 1                       # every slice mixes shifts from 1 on
        wt //= 32
        _run(oracle, x, wt, bias, mult, shift, stride, 0, 127)
        bias[c // 2] = 1 << 20                                # beyond the digits: the exact epilogue
        _run(oracle, x, wt, bias, mult, shift, stride, 0, 127)
    finally:
        binding.debug_dw_variant(0)


@pytest.mark.parametrize("stride", [1, 2])
def test_the_librarys_choice_for_a_large_layer(stride):
    """Large enough for the library to pick this kernel by itself: the same bytes as the CUDA-core one."""
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randint(-128, 128, (33, 57, 57, 144), generator=g, device="cuda", dtype=torch.int8)
    w = torch.randint(-128, 128, (144, 3, 3), generator=g, device="cuda", dtype=torch.int8)
    rq = binding.make_requant(torch.randint(-4096, 4097, (144,), generator=g, device="cuda", dtype=torch.int32),
                              torch.randint(1 << 30, (1 << 31) - 1, (144,), generator=g, device="cuda", dtype=torch.int32),
                              torch.randint(6, 12, (144,), generator=g, device="cuda", dtype=torch.int8))
    y = binding.dw_conv3x3_i8(x, w, rq, stride=stride)
    try:
        binding.debug_dw_variant(1)
        want = binding.dw_conv3x3_i8(x, w, rq, stride=stride)
    finally:
        binding.debug_dw_variant(0)
    assert torch.equal(y, want)
    assert binding.last_device_status() == binding.PROM_OK


@pytest.mark.parametrize("stride", [1, 2])
@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("b,h,w,c", [(1, 1, 1, 4), (1, 2, 3, 8), (2, 7, 7, 64), (1, 28, 28, 192), (9, 28, 30, 144)])
def test_units_of_the_cuda_core_kernel(oracle, stride, b, h, w, c, offset):
    """Small and large units on both sides of the rule, filters on a word boundary and one byte off it."""
    x, wt, bias, mult, shift = _case(47, b, h, w, c)
    store = torch.empty(c * 9 + 4, dtype=torch.int8, device="cuda")
    wd = store[offset:offset + c * 9].view(c, 3, 3)
    wd.copy_(torch.from_numpy(wt))
    try:
        binding.debug_dw_variant(1)
        for lo in (0, -128):
            rq = binding.make_requant(torch.from_numpy(bias).cuda(), torch.from_numpy(mult).cuda(), torch.from_numpy(shift).cuda(), lo, 127)
            y = binding.dw_conv3x3_i8(torch.from_numpy(x).cuda(), wd, rq, stride=stride)
            torch.cuda.synchronize()
            assert np.array_equal(y.cpu().numpy(), oracle.dw3x3(x, wt, bias, mult, shift, stride=stride, act_min=lo, act_max=127))
    finally:
        binding.debug_dw_variant(0)
