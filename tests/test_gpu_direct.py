"""Outputs that leave the tensor-core kernel straight from registers (subtiles of 32 to 256 columns over
permuted rows of B), byte for byte against the oracle: every split of a subtile into 64-column pieces and
a last one of 32, row counts around the 8-, 32- and 128-row steps, both fast epilogues, the exact one,
and the residual sum, with and without prepared operands."""
import numpy as np
import pytest
import torch

from paper_2505_03254_b200 import binding
from gpu_util import Guarded, make_case, oracle_y, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nt", [32, 64, 96, 128, 160, 192])
@pytest.mark.parametrize("m", [1, 7, 9, 33, 127, 129, 1000])
def test_every_subtile_width(oracle, m, nt):
    cin, cout = 48, 2 * nt
    x, lay = make_case(50 + m + nt, m, cin, cout)
    xd, wp, consts = to_device(x, lay)
    res = torch.from_numpy(np.random.default_rng(m).integers(-128, 128, size=(m, cout)).astype(np.int8))
    try:
        binding.debug_tc_plan_shape(m, cin, cout, nt=nt, fold=1)
        for lo, hi in ((0, 127), (-128, 127), (-5, 90)):
            want = oracle_y(oracle, x, lay, lo, hi)
            rq = binding.make_requant(*consts, lo, hi)
            for prepared in (False, True):
                g = Guarded(m * cout)
                if prepared:
                    ops = binding.pw_prepare(m, cin, wp, cout, rq)
                    binding.pw_conv_i8_prepared(xd, cout, ops, lo, hi, y=g.view(m, cout))
                else:
                    binding.pw_conv_i8(xd, wp, cout, rq, y=g.view(m, cout), variant="tc")
                g.check()
                assert np.array_equal(g.view(m, cout).cpu().numpy(), want), (lo, hi, prepared)
            g = Guarded(m * cout)
            binding.pw_conv_i8_res(xd, wp, cout, rq, res.cuda(), y=g.view(m, cout), variant="tc")
            g.check()
            assert np.array_equal(g.view(m, cout).cpu().numpy(), oracle.residual_add(want, res.numpy())), (lo, hi)
    finally:
        binding.debug_tc_plan_shape(m, cin, cout)
    assert binding.last_device_status() == binding.PROM_OK


def test_mixed_shifts_take_the_exact_epilogue(oracle):
    """A shift span above 4 leaves the one-multiply epilogue."""
    x, lay = make_case(77, 300, 64, 192, shift_lo=2, shift_hi=14)
    xd, wp, consts = to_device(x, lay)
    for lo in (0, -128):
        y = binding.pw_conv_i8(xd, wp, 192, binding.make_requant(*consts, lo, 127), variant="tc")
        torch.cuda.synchronize()
        assert np.array_equal(y.cpu().numpy(), oracle_y(oracle, x, lay, lo, 127))
