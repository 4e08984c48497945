"""An odd number of rows whose channel counts are 8 modulo 16: the automatic choice folds the rows in pairs
for TMA and takes the last row as a tile of its own.  Byte for byte against the oracle."""
import numpy as np
import pytest
import torch

from paper_2505_03254_b200 import binding, synth
from gpu_util import Guarded, make_case, oracle_y, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 3, 255, 257, 441, 1001, 12543])
@pytest.mark.parametrize("cin,cout", [(24, 144), (72, 432), (120, 720), (72, 24), (120, 240), (432, 72), (96, 264), (88, 88)])
def test_odd_rows(oracle, m, cin, cout):
    x, lay = make_case(9 + m, m, cin, cout)
    xd, wp, consts = to_device(x, lay)
    res = torch.from_numpy(np.random.default_rng(m).integers(-128, 128, size=(m, cout)).astype(np.int8))
    for lo in (0, -128):
        want = oracle_y(oracle, x, lay, lo, 127)
        rq = binding.make_requant(*consts, lo, 127)
        g = Guarded(m * cout)
        binding.pw_conv_i8(xd, wp, cout, rq, y=g.view(m, cout))
        g.check()
        assert np.array_equal(g.view(m, cout).cpu().numpy(), want)
        g = Guarded(m * cout)
        binding.pw_conv_i8_res(xd, wp, cout, rq, res.cuda(), y=g.view(m, cout))
        g.check()
        assert np.array_equal(g.view(m, cout).cpu().numpy(), oracle.residual_add(want, res.numpy()))
    assert binding.last_device_status() == binding.PROM_OK


def test_a_network_with_odd_rows(oracle):
    """Width 0.75 on 3 images of 48 x 48: the last layers have 27 rows of 72 and 120 channels."""
    table = synth.mobilenetv2_pointwise_layers(h0=48, w0=48, width=0.75)
    host, dev = [], []
    for i, l in enumerate(table):
        d = synth.make_layer(11, l.cin, l.cout, 0.5, index=i + 1)
        host.append(dict(cin=l.cin, cout=l.cout, in_stride=l.in_stride, w=d["w"].numpy(), bias=d["bias"].numpy(),
                         mult=d["mult"].numpy(), shift=d["shift"].numpy()))
        dev.append(dict(cin=l.cin, cout=l.cout, in_stride=l.in_stride, w_packed=binding.pack_ternary(d["w"].cuda()),
                        bias=d["bias"].cuda(), mult=d["mult"].cuda(), shift=d["shift"].cuda()))
    seq = binding.LayerSeq(dev)
    x0 = synth.act_post_relu6(11, (3, 48, 48, table[0].cin))
    ws = Guarded(seq.workspace_bytes(3, 48, 48), dtype=torch.uint8)
    y = binding.pw_layer_seq(seq, x0.cuda(), ws.t)
    ws.check("workspace")
    assert np.array_equal(y.cpu().numpy(), oracle.layer_seq(host, x0.numpy()))
    assert binding.last_device_status() == binding.PROM_OK
