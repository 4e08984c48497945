"""The row-resident kernel's operands in captured calls: each has its own, so that graphs captured on one stream may
run beside one another and beside calls on that stream, and those of a graph that is gone serve the next one."""
import pytest
import torch

from paper_2505_03254_b200 import binding
from gpu_util import make_case, to_device

pytestmark = pytest.mark.gpu

M, CIN, COUT = 148 * 100, 640, 512


def _layer(seed):
    x, lay = make_case(seed, M, CIN, COUT)
    xd, wp, consts = to_device(x, lay)
    rq = binding.make_requant(*consts)
    return xd, wp, rq, binding.pw_conv_i8(xd, wp, COUT, rq, variant="naive"), consts


def _capture(stream, layer, times=4):
    y = torch.empty((M, COUT), dtype=torch.int8, device="cuda")
    g = torch.cuda.CUDAGraph()
    before = binding.launch_count()
    with torch.cuda.graph(g, stream=stream):
        for _ in range(times):
            binding.pw_conv_i8(layer[0], layer[1], COUT, layer[2], y=y)
    assert binding.launch_count() - before == 2 * times          # operands and convolution: the row-resident kernel
    return g, y


def test_graphs_of_one_stream_run_at_the_same_time():
    home, others = torch.cuda.Stream(), [torch.cuda.Stream() for _ in range(2)]
    layers = [_layer(s) for s in (11, 12, 13)]
    torch.cuda.synchronize()
    graphs = [_capture(home, l) for l in layers[:2]]
    live = torch.empty((M, COUT), dtype=torch.int8, device="cuda")
    for _ in range(5):
        for _, y in graphs:
            y.fill_(-77)
        live.fill_(-77)
        torch.cuda.synchronize()
        for st, (g, _) in zip(others, graphs):
            with torch.cuda.stream(st):
                g.replay()
        with torch.cuda.stream(home):
            for _ in range(4):
                binding.pw_conv_i8(layers[2][0], layers[2][1], COUT, layers[2][2], y=live)
        torch.cuda.synchronize()
        for (_, y), l in zip(graphs, layers):
            assert torch.equal(y, l[3])
        assert torch.equal(live, layers[2][3])
    assert binding.last_device_status() == binding.PROM_OK


def test_memory_of_graphs_that_are_gone_is_used_again():
    home, layer = torch.cuda.Stream(), _layer(21)
    torch.cuda.synchronize()
    free = []
    for _ in range(12):
        g, y = _capture(home, layer)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, layer[3])
        g.reset()
        torch.cuda.synchronize()
        free.append(torch.cuda.mem_get_info()[0])
    # a graph's four buffers are 4 MB; its destruction may lag by a graph or two
    assert free[5] - free[-1] <= 2 * 4 * (1 << 20), free
