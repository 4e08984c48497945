"""The row-resident kernel over pairs of CTAs: row counts around its 256-row tiles (a second CTA with no rows, one
row, all but one), last column tiles of 32 to 256 columns, one and several units per pair, K up to its limit, and
the one-multiply epilogue for both clamps beside the 64-bit one."""
import numpy as np
import pytest

from paper_2505_03254_b200 import binding
from gpu_util import first_mismatch, make_case, run_variant, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lo,hi", [(0, 127), (-128, 127), (-7, 100)])
@pytest.mark.parametrize("m,cin,cout", [(1, 128, 64), (127, 640, 288), (128, 960, 272), (129, 576, 496), (255, 1024, 512),
                                        (257, 720, 240), (4999, 1024, 1280), (20225, 592, 336), (37889, 960, 144)])
def test_tiles_and_clamps(oracle, m, cin, cout, lo, hi):
    x, lay = make_case(m + cin + cout, m, cin, cout, 0.5, act="i8")
    xd, wp, consts = to_device(x, lay)
    binding.debug_tc_wide(2)
    try:
        y = run_variant(xd, wp, consts, cout, "tc", lo, hi)
    finally:
        binding.debug_tc_wide(0)
    assert binding.last_device_status() == binding.PROM_OK
    rows = np.unique(np.r_[0:min(m, 300), m // 2:min(m, m // 2 + 300), max(0, m - 300):m])
    want = oracle.conv_mul(x.numpy()[rows], lay["w"].numpy(), lay["bias"].numpy(), lay["mult"].numpy(), lay["shift"].numpy(), lo, hi)
    assert first_mismatch(np.asarray(y)[rows], want) is None
    # the rest against the plain kernel
    naive = run_variant(xd, wp, consts, cout, "naive", lo, hi)
    assert np.array_equal(np.asarray(y), np.asarray(naive))


@pytest.mark.parametrize("m,cin,cout,lo", [(12001, 320, 528, 0), (5921, 960, 320, -128), (3000, 592, 960, 0)])
def test_prepared(oracle, m, cin, cout, lo):
    """Operands prepared ahead where the library takes this kernel for them; another clamp than theirs is refused."""
    x, lay = make_case(m + cin, m, cin, cout, 0.5, act="i8")
    xd, wp, consts = to_device(x, lay)
    prep = binding.pw_prepare(m, cin, wp, cout, binding.make_requant(*consts, lo, 127))
    assert prep.numel() >= cout * cin                        # int8 weights: the row-resident form
    naive = run_variant(xd, wp, consts, cout, "naive", lo, 127)
    for _ in range(2):
        y = binding.pw_conv_i8_prepared(xd, cout, prep, lo, 127)
        assert np.array_equal(y.cpu().numpy(), np.asarray(naive))
    assert binding.last_device_status() == binding.PROM_OK
    y.fill_(-77)
    binding.pw_conv_i8_prepared(xd, cout, prep, -5, 90, y=y)
    assert binding.last_device_status() == binding.PROM_ERR_BAD_REQUANT
    assert bool((y == -77).all())
