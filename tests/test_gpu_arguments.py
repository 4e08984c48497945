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


def test_structures_of_another_type(layer):
    """What is read as constants, layers or jobs is one of the binding's structures, not any buffer of their size."""
    x, wp, rq = layer
    res = torch.zeros((M, COUT), dtype=torch.int8, device="cuda")
    x4, w9 = x.view(1, 16, 16, CIN), torch.zeros((CIN, 3, 3), dtype=torch.int8, device="cuda")
    for bad in (bytes(64), binding.PromLayer(), None):
        _refused(lambda: binding.pw_conv_i8(x, wp, COUT, bad), TypeError, "rq")
        _refused(lambda: binding.pw_conv_i8_res(x, wp, COUT, bad, res), TypeError, "rq")
        _refused(lambda: binding.dw_conv3x3_i8(x4, w9, bad), TypeError, "rq")
    seq = binding.LayerSeq([dict(cin=CIN, cout=COUT, in_stride=1, bias=torch.zeros(COUT, dtype=torch.int32, device="cuda"),
                                 mult=torch.full((COUT,), 1 << 30, dtype=torch.int32, device="cuda"),
                                 shift=torch.full((COUT,), 4, dtype=torch.int8, device="cuda"), w_packed=wp)])
    ws = torch.empty(max(1, seq.workspace_bytes(1, 16, 16)), dtype=torch.uint8, device="cuda")
    binding.pw_layer_seq(seq, x4, ws)
    layers, seq.array = seq.array, bytes(4096)
    _refused(lambda: binding.pw_layer_seq(seq, x4, ws), TypeError, "layers")
    seq.array = layers
    jobs = binding.QuantizeJobs([torch.ones((8, 16), device="cuda")])
    binding.quantize_ternary_batch(jobs=jobs)
    jobs.array = bytes(4096)
    _refused(lambda: binding.quantize_ternary_batch(jobs=jobs), TypeError, "jobs")
    assert binding.last_device_status() == binding.PROM_OK
