"""The weight quantiser's single comparison per weight against the binary64 definition, at the floats next to
the row's threshold and at the row lengths where the kernel changes its route."""
import numpy as np
import pytest
import torch

from paper_2505_03254_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cin", [4, 124, 128, 132, 1020, 1024, 1028, 1023, 4096])
def test_codes_next_to_the_threshold(oracle, cin):
    rng = np.random.default_rng(cin)
    w = (rng.standard_normal((12, cin)) * np.float32(10.0) ** rng.integers(-7, 6, size=(12, 1))).astype(np.float32)
    half = np.float32(0.5) * np.abs(w).astype(np.float64).mean(axis=1).astype(np.float32)
    for r in range(12):
        # neighbours of mean / 2 on both sides: the mean moves with them by less than a float's spacing
        # only now and then, so what decides is the oracle's own mean
        for i, steps in enumerate((-2, -1, 0, 1, 2)[: cin // 2]):
            v = half[r]
            for _ in range(abs(steps)):
                v = np.nextafter(v, np.float32(np.inf if steps > 0 else 0), dtype=np.float32)
            w[r, i] = v if r % 2 else -v
    q, alpha = oracle.quantize_ternary(w)
    packed, a = binding.quantize_ternary(torch.from_numpy(w).cuda())
    torch.cuda.synchronize()
    got, bad = oracle.unpack(packed.cpu().numpy(), 12, cin)
    assert bad == 0
    # binary64 sums in two orders agree to about cin * 2^-53: only a ratio that close to 1/2 may differ
    ratio = np.abs(w.astype(np.float64)) / np.maximum(alpha, 1e-5)[:, None]
    far = np.abs(ratio - 0.5) > cin * 2.0 ** -52
    assert far.mean() > 0.9 and np.array_equal(got[far], q[far])
    assert np.allclose(a.cpu().numpy(), alpha.astype(np.float32), rtol=1e-6, atol=0)
    assert binding.last_device_status() == binding.PROM_OK


def test_what_is_not_finite_is_reported():
    for bad in (float("nan"), float("inf"), float("-inf")):
        w = torch.ones((3, 64), device="cuda")
        w[1, 7] = bad
        binding.quantize_ternary(w)
        assert binding.last_device_status() == binding.PROM_ERR_BAD_WEIGHT


@pytest.mark.parametrize("cin", [63, 64, 2048])                 # row by element, held in registers, read twice
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
def test_a_row_that_is_not_finite_has_code_zero(cin, bad):
    w = torch.ones((3, cin), device="cuda")
    w[1, ::2] = -0.25
    w[1, 7] = bad
    packed, _ = binding.quantize_ternary(w)
    assert binding.last_device_status() == binding.PROM_ERR_BAD_WEIGHT
    one, _ = binding.quantize_ternary(torch.ones((1, cin), device="cuda"))
    packed, one = packed.view(3, -1), one.view(-1)
    assert bool((packed[1] == 0).all()) and torch.equal(packed[0], one) and torch.equal(packed[2], one)
