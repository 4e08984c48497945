"""Several threads that call the row-resident kernel on one stream: each call's operands reach its own convolution."""
import threading

import pytest
import torch

from paper_2505_03254_b200 import binding
from gpu_util import make_case, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("handle", ["shared", "per_thread_default"])
def test_threads_on_one_stream(handle):
    m, cin, cout, calls = 148 * 48, 640, 320, 60
    layers = []
    for seed in (1, 2, 3, 4):
        x, lay = make_case(seed, m, cin, cout)
        xd, wp, consts = to_device(x, lay)
        rq = binding.make_requant(*consts)
        layers.append((xd, wp, rq, binding.pw_conv_i8(xd, wp, cout, rq, variant="naive"), consts))
    torch.cuda.synchronize()
    # cudaStreamPerThread is the handle 2 in every thread
    stream = torch.cuda.Stream() if handle == "shared" else torch.cuda.ExternalStream(2)
    outs = [torch.empty((calls, m, cout), dtype=torch.int8, device="cuda") for _ in layers]
    torch.cuda.synchronize()
    start, failed = threading.Barrier(len(layers)), []

    def work(layer, out):
        try:
            start.wait()
            for k in range(calls):
                binding.pw_conv_i8(layer[0], layer[1], cout, layer[2], y=out[k], stream=stream)
        except Exception as e:
            failed.append(e)
    threads = [threading.Thread(target=work, args=a) for a in zip(layers, outs)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed, failed
    for layer, out in zip(layers, outs):
        assert bool((out == layer[3]).all())
    assert binding.last_device_status() == binding.PROM_OK
