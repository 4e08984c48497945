"""Calls overlap their set-up with the end of the kernel in front of them (programmatic dependent
launch): a call whose weights, constants or input the call before it has only just written must still
see them complete, in plain streams and in a captured graph."""
import pytest
import torch

from paper_2505_03254_b200 import binding, synth

pytestmark = pytest.mark.gpu


def _steps(m, k, n, pause):
    """Float weights are quantised into one buffer, over and over, each time read by the layer behind
    it, whose output the next layer and the depthwise layer read.  Returns every output."""
    dev = "cuda"
    g = torch.Generator(device=dev).manual_seed(m + k + n)
    x = synth.act_post_relu6(5, (m, k), device=dev)
    b1, m1, s1 = synth.requant_constants(6, n, device=dev)
    b2, m2, s2 = synth.requant_constants(7, k, device=dev)
    bias = torch.empty_like(b1)
    rq1, rq2 = binding.make_requant(bias, m1, s1), binding.make_requant(b2, m2, s2)
    w2 = binding.pack_ternary(synth.ternary_weights(8, k, n, device=dev))
    dw = synth.ternary_weights(9, k, 9, device=dev)
    floats = [torch.randn((n, k), generator=g, device=dev) for _ in range(12)]
    biases = [b1 + 37 * i for i in range(12)]
    packed = torch.empty((n, (k + 3) // 4), dtype=torch.uint8, device=dev)
    alpha = torch.empty((n,), device=dev)
    jobs = [binding.QuantizeJobs([w], out=[(packed, alpha)]) for w in floats]
    y1 = torch.empty((m, n), dtype=torch.int8, device=dev)
    y2 = torch.empty((m, k), dtype=torch.int8, device=dev)
    outs = [[torch.empty((m, n), dtype=torch.int8, device=dev), torch.empty((m, k), dtype=torch.int8, device=dev),
             torch.empty((m, k), dtype=torch.int8, device=dev)] for _ in floats]

    def step():
        for i in range(len(floats)):
            calls = (lambda: bias.copy_(biases[i]),
                     lambda: binding.quantize_ternary_batch(jobs=jobs[i]),
                     lambda: binding.pw_conv_i8(x, packed, n, rq1, y=y1),
                     lambda: binding.pw_conv_i8(y1, w2, k, rq2, y=y2),
                     lambda: binding.dw_conv3x3_i8(y2.view(1, m // 14, 14, k), dw, rq2, y=outs[i][2].view(1, m // 14, 14, k)),
                     lambda: outs[i][0].copy_(y1), lambda: outs[i][1].copy_(y2))
            for c in calls:
                c()
                if pause:
                    torch.cuda.synchronize()
    return step, outs


@pytest.mark.parametrize("m,k,n", [(196, 64, 384), (28, 32, 24), (28 * 896, 48, 96)])
def test_dependent_calls_see_each_other_complete(m, k, n):
    step, outs = _steps(m, k, n, pause=True)
    step()
    want = [t.clone() for o in outs for t in o]
    step, outs = _steps(m, k, n, pause=False)
    for _ in range(3):
        for o in outs:
            for t in o:
                t.fill_(-77)
        step()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(want, [t for o in outs for t in o]))
    side = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=side):
        step()
    for o in outs:
        for t in o:
            t.fill_(-77)
    graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(want, [t for o in outs for t in o]))
    assert binding.last_device_status() == binding.PROM_OK
