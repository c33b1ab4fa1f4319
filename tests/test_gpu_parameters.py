"""When parameters are read, and which layers a network may run behind others: everything against the CPU oracle, bit-exact."""
from __future__ import annotations

import copy

import numpy as np
import pytest

from paper_2011_10680_b200 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hq():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2011_10680_b200 import binding, build
    build.build()
    h = binding.Handle(0)
    yield h
    h.close()


def _table(bd, image_hw, classes=16):
    x = bd.avgpool(len(bd.layers) - 1)
    bd.conv(x, classes, 1, 1, 0, 8, relu=False, out_bits=32, op="linear")
    ids = range(len(bd.layers))
    return dict(layers=bd.layers, image_hw=image_hw, classes=classes, depth=0, conv_bits=[8], shapes=[bd.shape[i] for i in ids],
                bits=[bd.bits[i] for i in ids])


def _builder(seed, image_hw):
    bd = inputs._Builder(seed)
    bd.scale[-1], bd.shape[-1], bd.bits[-1] = 2.0 ** -4, (image_hw, image_hw, 3), 8
    return bd


def test_int32_add_behind_a_convolution_of_short_rows(hq):
    """16-channel 3x3 convolutions in front of INT32 adds: the direct kernel declines them (their patch matrix is cheaper),
    so the add does not run behind them."""
    from test_gpu_parity import run_network_and_compare
    run_network_and_compare(hq, inputs.resnet_table(18, seed=12, image_hw=64, classes=24, width=16, int32_stream=True), batch=2, seed=3)


def test_a_clamp_outside_its_type_is_refused_behind_an_int32_add(hq):
    """A REQUANT layer whose clamp leaves the 8-bit range is refused whether it runs alone or behind the add before it."""
    from paper_2011_10680_b200 import binding
    t = inputs.resnet_table(50, seed=8, image_hw=64, classes=24, width=32, int32_stream=True)
    layer = next(l for l in t["layers"] if l["op"] == "requant" and t["layers"][l["in0"]]["op"] == "add")
    images = binding.to_device(inputs.random_images(4, 2, 64))
    for qmin, qmax, want in ((0, 255, binding.HQ_OK), (0, 256, binding.HQ_ERR_INVALID_ARG), (-1, 255, binding.HQ_ERR_INVALID_ARG),
                             (9, 8, binding.HQ_ERR_INVALID_ARG)):
        layer["qmin"], layer["qmax"] = qmin, qmax
        net = binding.Network(hq, t, 2)
        try:
            logits = binding.alloc_out(*net.logits_shape, 32, 1)
            assert net.run(images, logits, net.alloc_taps()) == want
            with torch.cuda.stream(torch.cuda.Stream()):
                assert net.run(images, logits, None) == want
                hq.sync()
        finally:
            net.close()


def _rewrite_and_compare(hq, table, batch, change):
    """Run a network, overwrite the parameters of some layers in place, run it again: the new values count."""
    from oracle.network import run_network
    from paper_2011_10680_b200 import binding
    images = inputs.random_images(21, batch, table["image_hw"])
    changed = copy.deepcopy(table)
    change(changed["layers"])
    want = [run_network(t, images)[-1] for t in (table, changed)]
    assert not np.array_equal(*want)
    net, other = binding.Network(hq, table, batch), binding.Network(hq, changed, batch)
    try:
        d_img = binding.to_device(images)
        logits = binding.alloc_out(*net.logits_shape, 32, 1)
        with torch.cuda.stream(torch.cuda.Stream()):
            for ref in want:
                assert net.run(d_img, logits, None) == binding.HQ_OK
                hq.sync()
                assert np.array_equal(logits.cpu().numpy().reshape(ref.shape), ref)
                for mine, theirs in zip(net._keep, other._keep):
                    for key, tensor in mine.items():
                        if tensor is not None:
                            tensor.copy_(theirs[key])
                torch.cuda.synchronize()
        net.check_guards()
    finally:
        net.close()
        other.close()


@pytest.mark.parametrize("hw,batch", [(56, 11), (26, 41)])
def test_pixel_pair_layers_follow_their_parameters(hq, hw, batch):
    """3x3 layers over 64 channels in the pixel-pair form of a network: weights, bias and pairs are read at every run."""
    bd = _builder(hw, 2 * hw)
    x = bd.conv(-1, 64, 3, 2, 1, 8, relu=True, out_bits=8)
    bd.conv(x, 64, 3, 1, 1, 8, relu=True, out_bits=8)

    def change(layers):
        l = layers[1]
        l["wgt"], l["bias"], l["b"], l["c"] = np.ascontiguousarray(l["wgt"][::-1]), l["bias"][::-1].copy(), np.roll(l["b"], 1), np.roll(l["c"], 1)
    _rewrite_and_compare(hq, _table(bd, 2 * hw), batch, change)


@pytest.mark.parametrize("batch", [2, 21])
@pytest.mark.parametrize("shifts", [None, (45, 8)])
def test_concatenations_follow_their_pairs(hq, batch, shifts):
    """The pairs of a concatenation's branches are read at every run, below and above the size that works with narrow pairs;
    from a pair that scales everything to zero to one with the same multiplier and the smallest shift without a narrow form."""
    bd = _builder(41, 42)
    x = bd.conv(-1, 48, 3, 1, 0, 8, relu=True, out_bits=8)
    cat = bd.concat([bd.conv(x, 80, 1, 1, 0, 8, relu=True, out_bits=8), x])
    if shifts:
        for c in bd.layers[cat]["cs"]:
            c[::2] = shifts[0]

    def change(layers):
        if shifts:
            for c in layers[cat]["cs"]:
                c[::2] = shifts[1]
            return
        layers[cat]["bs"] = [np.roll(b, 3) for b in layers[cat]["bs"]]
        layers[cat]["cs"] = [c + 1 for c in layers[cat]["cs"]]
    _rewrite_and_compare(hq, _table(bd, 42), batch, change)


@pytest.mark.parametrize("writer", ["library", "torch"])
@pytest.mark.parametrize("cfg", [
    # path, n, hw, cin, cout, k, bits, residual
    (2, 4, 28, 64, 128, 3, 8, False),      # resident weights
    (3, 8, 28, 64, 64, 3, 8, False),       # the same in strips
    (2, 49, 28, 64, 256, 1, 8, True),      # residual through tensor memory
    (2, 13, 14, 256, 256, 3, 8, False),    # weights that travel with the stages
    (3, 8, 28, 64, 64, 3, 4, False),       # packed operands, widened in the launch before, in strips
    (2, 4, 28, 64, 128, 3, 4, True),       # ... and in resident blocks
    (0, 3, 17, 3, 32, 3, 8, False),        # patch matrix
    (4, 1, 14, 64, 64, 3, 8, False),       # the kernel for small problems
    (4, 1, 14, 64, 64, 3, 4, True),
])
def test_single_calls_follow_parameters_written_just_before(hq, cfg, writer):
    """Weights, bias and pairs that the launch right before a call on the same stream has written, by an element-wise call of
    the library (whose launch lets the next one start early) or by a copy kernel: no call may read them before it ended."""
    from oracle import hqref
    from paper_2011_10680_b200 import binding
    path, n, hw, cin, cout, k, bits, residual = cfg
    cases = [inputs.conv_case(700 + i, n, hw, hw, cin, cout, k, 1, k // 2, bits=bits, residual=residual, c_range=(39, 44)) for i in range(4)]
    for case in cases:                     # one set of activations, four sets of parameters
        case["x"], case["res"] = cases[0]["x"], cases[0]["res"]
    dev = binding.upload_case(cases[0])
    names = [f for f in ("wgt", "bias", "b", "c", "rb", "rc") if dev[f] is not None]
    one = torch.full((max(cin, cout),), 1 << 30, dtype=torch.int32, device="cuda")
    thirty = torch.full_like(one, 30)      # dn(v, 2^30, 30) = v
    sources = []
    for case in cases:
        src = {f: binding.to_device(case[f]) for f in names}
        if writer == "library":            # weights as one signed byte per value
            w = case["wgt"] if bits == 8 else inputs.unpack4(case["wgt"], True).astype(np.int8)
            src["wgt"] = binding.to_device(np.ascontiguousarray(w))
        sources.append(src)

    def write(src, f):
        if writer == "torch":
            dev[f].copy_(src[f])
        elif f == "wgt":
            lo, hi = (-128, 127) if bits == 8 else (-8, 7)
            st = hq.residual_add(src[f], 8, 1, one, thirty, None, 0, 0, None, None, cin, 0, lo, hi, dev[f], bits, 1)
            assert st == binding.HQ_OK, binding.status_string(st)
        else:
            shape = (1, 1, 1, cout)
            st = hq.residual_add(src[f].view(shape), 32, 1, one, thirty, None, 0, 0, None, None, cout, 0, -(1 << 31), (1 << 31) - 1,
                                 dev[f].view(shape), 32, 1)
            assert st == binding.HQ_OK, binding.status_string(st)

    refs = [hqref.conv_case(case) for case in cases]
    outs = [binding.alloc_out(cases[0]["n"], cases[0]["ho"], cases[0]["wo"], cout, 8, cases[0]["out_signed"]) for _ in range(4 * len(names))]
    hq.set_conv_path(path)
    try:
        # every parameter in turn is the last one written before the call
        for r, last in enumerate(names):
            for i, src in enumerate(sources):
                for f in names:
                    if f != last:
                        write(src, f)
                write(src, last)
                st, _ = hq.conv_case(cases[0], dev, outs[4 * r + i])
                assert st == binding.HQ_OK, binding.status_string(st)
        hq.sync()
    finally:
        hq.set_conv_path(0)
    for r, last in enumerate(names):
        for i, ref in enumerate(refs):
            got = outs[4 * r + i].cpu().numpy().view(ref.dtype).reshape(ref.shape)
            assert np.array_equal(got, ref), (last, i, int((got != ref).sum()), ref.size)
