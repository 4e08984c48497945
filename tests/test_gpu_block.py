"""A block of a sequence (expand, depthwise 3x3, project with its skip connection) in one launch: bytes equal
to the oracle's at the edges of its bands, units, slices, rings and clusters."""
import numpy as np
import pytest
import torch

from paper_2505_03254_b200 import binding, synth
from gpu_util import Guarded

pytestmark = pytest.mark.gpu


def _layer(rng, seed, cin, cout, stride=1, **kw):
    d = synth.make_layer(seed, cin, cout, 0.5)
    h = dict(cin=cin, cout=cout, in_stride=stride, w=d["w"].numpy(), bias=d["bias"].numpy(), mult=d["mult"].numpy(),
             shift=d["shift"].numpy(), act_min=kw.get("act_min", 0), skip=kw.get("skip", False))
    if "shift" in kw:
        h["shift"] = kw["shift"].astype(np.int8)
    if kw.get("dw"):
        h["dw_w"] = rng.integers(-128, 128, size=(cin, 3, 3)).astype(np.int8)
        h["dw_bias"] = rng.integers(-3000, 3001, size=cin).astype(np.int32)
        h["dw_mult"] = rng.integers(1 << 30, (1 << 31) - 1, size=cin).astype(np.int32)
        h["dw_shift"] = rng.integers(*kw.get("dw_shift", (8, 11)), size=cin).astype(np.int8)
    dev = {k: v for k, v in h.items() if k not in ("w", "skip")}
    dev = {k: torch.from_numpy(v).cuda() if isinstance(v, np.ndarray) else v for k, v in dev.items()}
    dev["w_packed"] = binding.pack_ternary(d["w"].cuda())
    dev["add_block_input"] = h["skip"]
    return h, dev


def _want(oracle, e, q, x):
    b, h, w, c = x.shape
    t = oracle.conv_mul(x.reshape(-1, c), e["w"], e["bias"], e["mult"], e["shift"], e["act_min"], 127).reshape(b, h, w, -1)
    t = oracle.dw3x3(t, q["dw_w"], q["dw_bias"], q["dw_mult"], q["dw_shift"], stride=q["in_stride"], act_min=0, act_max=127)
    b, h, w, c = t.shape
    y = oracle.conv_mul(t.reshape(-1, c), q["w"], q["bias"], q["mult"], q["shift"], q["act_min"], 127).reshape(b, h, w, -1)
    return oracle.residual_add(y, x) if q["skip"] else y


def _want_sequence(oracle, layers, x):
    """One layer after the other; a skip connection adds the input of the layer before."""
    before = None
    for l in layers:
        t = x
        if "dw_w" in l:
            t = oracle.dw3x3(x, l["dw_w"], l["dw_bias"], l["dw_mult"], l["dw_shift"], stride=l["in_stride"], act_min=0, act_max=127)
        b, h, w, c = t.shape
        y = oracle.conv_mul(t.reshape(-1, c), l["w"], l["bias"], l["mult"], l["shift"], l["act_min"], 127).reshape(b, h, w, -1)
        before, x = x, oracle.residual_add(y, before) if l["skip"] else y
    return x


def _run(dev, x, rows=0, split=0, mode=2):
    binding.debug_seq_block(mode, rows, split)
    try:
        seq = binding.LayerSeq(dev)
        b, h, w, _ = x.shape
        fused = binding.debug_layer_seq_output_offset(seq, b, h, w, 0)[0] == -2
        ws = Guarded(seq.workspace_bytes(b, h, w), dtype=torch.uint8, fill=0)
        s = seq.total_stride
        y = Guarded(b * (h // s) * (w // s) * dev[-1]["cout"])
        binding.pw_layer_seq(seq, x, ws.t, y.view(b, h // s, w // s, dev[-1]["cout"]))
        ws.check("workspace"); y.check("output")
        assert binding.last_device_status() == binding.PROM_OK
        return y.view(b, h // s, w // s, dev[-1]["cout"]).cpu().numpy(), fused
    finally:
        binding.debug_seq_block()


CASES = [
    # batch, h, w, cin, expanded, cout, stride, skip, rows, split
    (1, 7, 7, 160, 960, 160, 1, True, 0, 0),
    (5, 7, 7, 160, 960, 320, 1, False, 0, 8),          # two images per item, project sums of 320 columns
    (3, 14, 14, 64, 384, 64, 1, True, 7, 1),
    (2, 14, 14, 72, 432, 72, 1, True, 0, 3),           # channel counts that are 8 modulo 16, a half-empty last slice
    (2, 14, 14, 96, 576, 160, 2, False, 0, 0),
    (2, 28, 28, 32, 192, 32, 1, True, 5, 1),           # a ragged last band
    (3, 28, 20, 32, 192, 64, 2, False, 3, 2),
    (2, 56, 56, 24, 144, 24, 1, True, 0, 0),
    (1, 56, 56, 24, 144, 32, 2, False, 4, 1),
    (1, 112, 112, 16, 96, 24, 2, False, 2, 1),
    (1, 5, 3, 8, 72, 8, 1, False, 1, 2),               # one row per band, planes of a few pixels
    (4, 2, 2, 8, 32, 16, 2, False, 0, 0),
    (1, 1, 1, 16, 96, 24, 1, False, 0, 0),
    (40, 14, 14, 16, 64, 16, 1, True, 2, 1),           # more items than CTAs: several per CTA
    (700, 7, 7, 16, 32, 16, 1, True, 0, 1),            # ... of one slice each
    (9, 10, 6, 24, 96, 48, 1, False, 0, 2),
    (2, 16, 30, 24, 96, 80, 1, False, 16, 1),          # sums that end with tensor memory
    (2, 16, 30, 24, 96, 72, 1, False, 16, 2),
    (2, 30, 30, 16, 96, 16, 1, True, 30, 2),
]


@pytest.mark.parametrize("b,h,w,cin,mid,cout,stride,skip,rows,split", CASES)
def test_block(oracle, b, h, w, cin, mid, cout, stride, skip, rows, split):
    rng = np.random.default_rng(b * 1000 + h * 10 + cin)
    e, de = _layer(rng, 3, cin, mid)
    q, dq = _layer(rng, 4, mid, cout, stride, dw=True, act_min=-128, skip=skip)
    x = synth.act_post_relu6(9 + h, (b, h, w, cin))
    got, fused = _run([de, dq], x.cuda(), rows, split)
    assert fused
    assert np.array_equal(got, _want(oracle, e, q, x.numpy()))


@pytest.mark.parametrize("p_clamp", [(-128, 127), (-128, 60), (-30, 60)])
@pytest.mark.parametrize("e_clamp,d_clamp,fused", [((0, 127), (0, 127), True), ((-128, 127), (0, 127), False), ((0, 100), (0, 127), False),
                                                   ((0, 127), (-128, 127), False), ((0, 127), (0, 100), False), ((1, 127), (5, 127), False)])
def test_clamps_that_the_library_takes_as_a_block(oracle, e_clamp, d_clamp, fused, p_clamp):
    rng = np.random.default_rng(41)
    e, de = _layer(rng, 43, 32, 192)
    q, dq = _layer(rng, 44, 192, 32, dw=True, act_min=-128, skip=True)
    x = synth.act_post_relu6(45, (16, 28, 28, 32))
    seq = binding.LayerSeq([de, dq])
    seq.array[0].rq.act_min, seq.array[0].rq.act_max = e_clamp
    seq.array[1].dw_rq.act_min, seq.array[1].dw_rq.act_max = d_clamp
    seq.array[1].rq.act_min, seq.array[1].rq.act_max = p_clamp
    t = oracle.conv_mul(x.numpy().reshape(-1, 32), e["w"], e["bias"], e["mult"], e["shift"], *e_clamp).reshape(16, 28, 28, 192)
    t = oracle.dw3x3(t, q["dw_w"], q["dw_bias"], q["dw_mult"], q["dw_shift"], stride=1, act_min=d_clamp[0], act_max=d_clamp[1])
    y = oracle.conv_mul(t.reshape(-1, 192), q["w"], q["bias"], q["mult"], q["shift"], *p_clamp).reshape(x.shape)
    want = oracle.residual_add(y, x.numpy())
    for mode in (0, 2):                                 # by the library's rule, and wherever possible
        binding.debug_seq_block(mode)
        try:
            taken = binding.debug_layer_seq_output_offset(seq, 16, 28, 28, 0)[0] == -2
            got = binding.pw_layer_seq(seq, x.cuda(), torch.empty((seq.workspace_bytes(16, 28, 28),), dtype=torch.uint8, device="cuda"))
            assert np.array_equal(got.cpu().numpy(), want), mode
        finally:
            binding.debug_seq_block()
        assert taken == (fused or mode == 2)
    assert binding.last_device_status() == binding.PROM_OK


@pytest.mark.parametrize("b,h,w,cin,mid,cout,stride,blocks,taken", [
    (16, 28, 28, 32, 192, 32, 1, 1, True),
    (2, 20, 20, 32, 192, 32, 1, 1, False),             # 13.6 us against 11.7
    (2, 33, 9, 184, 672, 200, 1, 1, False),            # 20.5 against 16.4
    (149, 10, 10, 256, 200, 112, 1, 1, False),         # 32.9 against 23.8: wide inputs, two items per CTA
    (64, 14, 14, 64, 384, 64, 1, 1, True),
    (58, 20, 20, 232, 32, 232, 1, 3, False),
    (9, 28, 28, 24, 144, 24, 1, 3, True),
])
def test_blocks_that_the_library_takes(b, h, w, cin, mid, cout, stride, blocks, taken):
    """By the rule: blocks that save too little in their call have one launch per layer."""
    rng = np.random.default_rng(47)
    dev = []
    for i in range(blocks):
        dev += [_layer(rng, 48, cin, mid)[1], _layer(rng, 49, mid, cout, stride, dw=True, act_min=-128)[1]]
    seq = binding.LayerSeq(dev)
    got = [binding.debug_layer_seq_output_offset(seq, b, h, w, 2 * i)[0] == -2 for i in range(blocks)]
    assert got == [taken] * blocks


@pytest.mark.parametrize("cin,mid,cout", [(24, 72, 24), (64, 192, 40)])
@pytest.mark.parametrize("what", ["expand", "depthwise", "both"])
def test_block_with_constants_far_apart(oracle, what, cin, mid, cout):
    """Shifts, multipliers and biases at the ends of their documented ranges beside ordinary ones of the same slice."""
    rng = np.random.default_rng(mid)
    e, de = _layer(rng, 35, cin, mid)
    q, dq = _layer(rng, 36, mid, cout, dw=True, act_min=-128, skip=cin == cout)
    for h, dev, pre, mine in ((e, de, "", what != "depthwise"), (q, dq, "dw_", what != "expand")):
        if not mine:
            continue
        for name, values in (("shift", [0, 1, 15, 30, 31]), ("mult", [0, 1, 1 << 30, (1 << 31) - 1]),
                             ("bias", [-(1 << 28), -(1 << 20), 467000, 1 << 20, 1 << 28])):
            a = h[pre + name].copy()
            at = rng.random(mid) < 0.2
            a[at] = rng.choice(values, size=int(at.sum()))
            h[pre + name] = a
            dev[pre + name] = torch.from_numpy(a).cuda()
    x = synth.act_post_relu6(37, (3, 14, 14, cin))
    got, fused = _run([de, dq], x.cuda())
    assert fused
    assert np.array_equal(got, _want(oracle, e, q, x.numpy()))


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("third", ["pointwise", "depthwise", "more_behind"])
def test_skip_connection_behind_a_block(oracle, third, mode):
    """A layer that adds the expanded tensor of the two layers in front of it: that tensor has to be written."""
    rng = np.random.default_rng(23)
    b, side, cin, mid = 64, 14, 64, 384
    layers = [_layer(rng, 11, cin, mid), _layer(rng, 12, mid, cin, dw=True, act_min=-128, skip=True),
              _layer(rng, 13, cin, mid, skip=True, dw=third == "depthwise")]
    if third == "more_behind":
        layers += [_layer(rng, 14, mid, cin, dw=True, act_min=-128), _layer(rng, 15, cin, mid),
                   _layer(rng, 16, mid, cin, dw=True, act_min=-128, skip=True)]
    host, dev = [h for h, _ in layers], [d for _, d in layers]
    x = synth.act_post_relu6(31, (b, side, side, cin))
    binding.debug_seq_block(mode)
    try:
        pair = binding.LayerSeq(dev[:2])
        assert binding.debug_layer_seq_output_offset(pair, b, side, side, 0)[0] == -2      # a block, on its own
        seq = binding.LayerSeq(dev)
        offsets = [binding.debug_layer_seq_output_offset(seq, b, side, side, i)[0] for i in range(len(dev) - 1)]
    finally:
        binding.debug_seq_block()
    assert [i for i, o in enumerate(offsets) if o == -2] == ([4] if third == "more_behind" else [])
    xg = Guarded(x.numel())
    xg.t.copy_(x.reshape(-1))
    got, _ = _run(dev, xg.view(*x.shape), mode=mode)
    assert np.array_equal(got, _want_sequence(oracle, host, x.numpy()))


@pytest.mark.parametrize("what", ["wide_shifts", "signed_expand", "dw_shift_0", "clamped_project"])
def test_block_exact_epilogues(oracle, what):
    """Constants and clamps that the one-multiply epilogues do not take."""
    rng = np.random.default_rng(17)
    cin, mid, cout = 24, 72, 24
    kw = {}
    if what == "wide_shifts":
        kw["shift"] = rng.integers(6, 14, size=mid)
    if what == "signed_expand":
        kw["act_min"] = -128
    e, de = _layer(rng, 5, cin, mid, **kw)
    q, dq = _layer(rng, 6, mid, cout, dw=True, skip=True, act_min=-20 if what == "clamped_project" else -128,
                   dw_shift=(0, 14) if what == "dw_shift_0" else (8, 11))
    x = synth.act_post_relu6(2, (3, 14, 14, cin))
    got, fused = _run([de, dq], x.cuda())
    assert fused
    assert np.array_equal(got, _want(oracle, e, q, x.numpy()))


@pytest.mark.parametrize("split", [1, 3])
@pytest.mark.parametrize("layer,name,value", [(0, "mult", -1), (1, "dw_bias", (1 << 28) + 1), (1, "shift", 32)])
def test_block_with_bad_constants(layer, name, value, split):
    """A constant out of range in any of the block's layers, one channel of one slice: reported, and no output written."""
    rng = np.random.default_rng(29)
    dev = [_layer(rng, 9, 32, 192)[1], _layer(rng, 10, 192, 32, dw=True, act_min=-128, skip=True)[1]]
    x = synth.act_post_relu6(5, (3, 14, 14, 32)).cuda()
    for channel in (0, dev[layer][name].numel() - 1):
        was = dev[layer][name][channel].item()
        dev[layer][name][channel] = value
        binding.debug_seq_block(2, 5, split)
        try:
            seq = binding.LayerSeq(dev)
            assert binding.debug_layer_seq_output_offset(seq, 3, 14, 14, 0)[0] == -2
            y = Guarded(x.numel())
            binding.pw_layer_seq(seq, x, torch.empty((seq.workspace_bytes(3, 14, 14),), dtype=torch.uint8, device="cuda"), y.view(*x.shape))
        finally:
            binding.debug_seq_block()
        assert binding.last_device_status() == binding.PROM_ERR_BAD_REQUANT
        y.check("output")
        assert bool((y.t == -77).all()), (channel, split)
        dev[layer][name][channel] = was
    got, fused = _run(dev, x, 5, split)
    assert fused and (got != -77).any()


@pytest.mark.parametrize("layer", [0, 1])
def test_block_with_an_invalid_weight_code(layer):
    rng = np.random.default_rng(31)
    dev = [_layer(rng, 9, 32, 192)[1], _layer(rng, 10, 192, 32, dw=True, act_min=-128)[1]]
    dev[layer]["w_packed"][-1, -1] = 0b10000000           # code 10 in the last place of the last row
    binding.debug_seq_block(2)
    try:
        seq = binding.LayerSeq(dev)
        assert binding.debug_layer_seq_output_offset(seq, 2, 14, 14, 0)[0] == -2
        x = synth.act_post_relu6(5, (2, 14, 14, 32)).cuda()
        binding.pw_layer_seq(seq, x, torch.empty((seq.workspace_bytes(2, 14, 14),), dtype=torch.uint8, device="cuda"))
    finally:
        binding.debug_seq_block()
    assert binding.last_device_status() == binding.PROM_ERR_BAD_WEIGHT


def _mixed(rng):
    """Blocks between layers that are none: a depthwise + project layer without an expanding one, twice, and a last pointwise layer."""
    return [_layer(rng, 51, 32, 32, dw=True, act_min=-128), _layer(rng, 52, 32, 192), _layer(rng, 53, 192, 32, dw=True, act_min=-128, skip=True),
            _layer(rng, 54, 32, 48, dw=True, act_min=-128), _layer(rng, 55, 48, 288), _layer(rng, 56, 288, 64, 2, dw=True, act_min=-128),
            _layer(rng, 57, 64, 96)]


def test_block_falls_back(oracle):
    """A workspace without room for the blocks' operands: one launch per layer in the regions of that layout, the same bytes,
    and the same least size as without blocks."""
    # (few pixels: the operands then outweigh the expanded tensors that need no room)
    layers = _mixed(np.random.default_rng(19))
    host, dev = [h for h, _ in layers], [d for _, d in layers]
    x = synth.act_post_relu6(3, (1, 6, 6, 32))
    want = _want_sequence(oracle, host, x.numpy())
    seq, xd = binding.LayerSeq(dev), x.cuda()

    def call(nbytes):
        ws = Guarded(nbytes, dtype=torch.uint8, fill=0x33)
        y = Guarded(want.size)
        before = binding.launch_count()
        binding.pw_layer_seq(seq, xd, ws.t, y.view(*want.shape))
        launches = binding.launch_count() - before
        ws.check("workspace"); y.check("output")
        assert np.array_equal(y.view(*want.shape).cpu().numpy(), want), nbytes
        return launches

    def least():                                        # the smallest workspace that is not refused
        lo, hi = 0, 1 << 22
        while lo + 16 < hi:
            mid = (lo + hi) // 32 * 16
            try:
                call(mid)
                hi = mid
            except binding.PromError as err:
                assert err.code == binding.PROM_ERR_WORKSPACE
                lo = mid
        return hi

    binding.debug_seq_block(1)
    try:
        plain, least_plain = seq.workspace_bytes(1, 6, 6), least()
        one_per_layer = call(plain)
    finally:
        binding.debug_seq_block()
    binding.debug_seq_block(2)
    try:
        need = seq.workspace_bytes(1, 6, 6)
        assert [binding.debug_layer_seq_output_offset(seq, 1, 6, 6, i)[0] == -2 for i in range(6)] == [False, True, False, False, True, False]
        assert need > plain
        assert call(need) == one_per_layer - 4 + 1      # two launches fewer per block, one more for their operands
        assert call(plain) == one_per_layer and call(need - 1) == one_per_layer
        assert least() == least_plain
    finally:
        binding.debug_seq_block()
    assert binding.last_device_status() == binding.PROM_OK


def test_block_with_an_output_that_overlaps_its_input(oracle):
    rng = np.random.default_rng(19)
    e, de = _layer(rng, 7, 32, 192)
    q, dq = _layer(rng, 8, 192, 32, dw=True, act_min=-128, skip=True)
    x = synth.act_post_relu6(3, (2, 14, 14, 32))
    binding.debug_seq_block(2)
    try:
        seq = binding.LayerSeq([de, dq])
        ws = torch.empty((seq.workspace_bytes(2, 14, 14),), dtype=torch.uint8, device="cuda")
        before = binding.launch_count()
        y = binding.pw_layer_seq(seq, x.cuda(), ws)
        fused = binding.launch_count() - before
        xy = x.cuda()
        before = binding.launch_count()
        binding.pw_layer_seq(seq, xy, ws, xy)
        assert binding.launch_count() - before > fused
    finally:
        binding.debug_seq_block()
    torch.cuda.synchronize()
    want = _want(oracle, e, q, x.numpy())
    assert np.array_equal(y.cpu().numpy(), want) and np.array_equal(xy.cpu().numpy(), want)


@pytest.mark.parametrize("seed", range(6))
def test_random_blocks_match_one_launch_per_layer(seed):
    """Sequences of random blocks (odd planes, any multiple of 8 channels, both strides, ordinary and other clamps on each of the
    three layers), in whatever geometry the planner takes, live and from a captured graph: the bytes of one launch per layer."""
    rng = np.random.default_rng(100 + seed)
    pairs = taken = most = 0
    for _ in range(4):
        b = int(rng.integers(1, 12)) if rng.random() < 0.8 else int(rng.integers(150, 320))
        h, w = int(rng.integers(1, 40)), int(rng.integers(1, 40))
        cin, dev, clamps = 8 * int(rng.integers(1, 25)), [], []
        x = synth.act_post_relu6(seed, (b, h, w, cin)).cuda()
        n = int(rng.integers(1, 4))
        for i in range(n):
            stride = 2 if h % 2 == 0 and w % 2 == 0 and rng.random() < 0.4 else 1
            mid = 8 * int(rng.integers(4, 90))
            skip = stride == 1 and rng.random() < 0.5
            cout = cin if skip else 8 * int(rng.integers(1, 40))
            fast = rng.random() < 0.7
            _, e = _layer(rng, seed * 10 + i, cin, mid)
            _, q = _layer(rng, seed * 10 + i + 5, mid, cout, stride, dw=True, skip=skip, dw_shift=(8, 11) if fast else (0, 14))
            dev += [e, q]
            clamps += [[(0, 127)] if fast else [(-128, 127), (0, 101), (-60, 55)], [(0, 127)] if fast else [(-128, 90), (0, 127), (3, 127)],
                       [(-128, 127), (-40, 127), (-128, 70), (0, 127)]]
            h, w, cin = h // stride, w // stride, cout
        seq = binding.LayerSeq(dev)
        for i in range(n):
            for rq, of in ((seq.array[2 * i].rq, 0), (seq.array[2 * i + 1].dw_rq, 1), (seq.array[2 * i + 1].rq, 2)):
                choice = clamps[3 * i + of]
                rq.act_min, rq.act_max = choice[int(rng.integers(len(choice)))]
        shape = (b, h, w, cin)
        out = {}
        for mode in (1, 2):
            binding.debug_seq_block(mode)
            try:
                ws = Guarded(seq.workspace_bytes(*x.shape[:3]), dtype=torch.uint8, fill=0)
                y = Guarded(int(np.prod(shape)))
                fused = [binding.debug_layer_seq_output_offset(seq, *x.shape[:3], 2 * i)[0] == -2 for i in range(n)]
                binding.pw_layer_seq(seq, x, ws.t, y.view(*shape))
                ws.check("workspace"); y.check("output")
                out[mode] = y.t.cpu().numpy()
                if mode == 1:
                    assert not any(fused)
                    continue
                pairs += n; taken += sum(fused); most = max(most, sum(fused))
                y.t.fill_(-77)
                s = torch.cuda.Stream()
                with torch.cuda.stream(s):
                    g = torch.cuda.CUDAGraph()
                    with torch.cuda.graph(g, stream=s):
                        binding.pw_layer_seq(seq, x, ws.t, y.view(*shape))
                        binding.pw_layer_seq(seq, x, ws.t, y.view(*shape))
                g.replay()
                ws.check("workspace"); y.check("output")
                assert np.array_equal(y.t.cpu().numpy(), out[1])
            finally:
                binding.debug_seq_block()
        assert np.array_equal(out[2], out[1]), (x.shape, [(d["cin"], d["cout"], d["in_stride"]) for d in dev], fused)
        assert binding.last_device_status() == binding.PROM_OK
    assert 2 * taken >= pairs and most >= 2, (taken, pairs, most)
