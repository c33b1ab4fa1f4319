"""The one-tile-per-CTA convolution kernel (small problems) against the CPU oracle, bit-exact, forced by conv path 4."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2011_10680_b200 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [
    # n, h, w, cin, cout, k, stride, pad, bits, out_bits, residual bits (0: none), relu
    (1, 7, 7, 512, 512, 3, 1, 1, 8, 8, 0, True),      # 49 pixels, 36 K blocks: clusters of eight CTAs, ragged split
    (1, 1, 1, 2048, 1000, 1, 1, 0, 8, 32, 0, False),  # one pixel (16-pixel tile), INT32 result, ragged channel tile
    (3, 5, 5, 64, 256, 1, 1, 0, 8, 8, 8, True),       # 75 pixels: a full tile and a remainder, 8-bit residual words
    (2, 9, 4, 48, 100, 3, 2, 1, 8, 8, 32, False),     # cin not a multiple of 32, INT32 residual, signed output
    (1, 6, 5, 16, 30, 5, 1, 2, 8, 8, 8, True),        # 30 pixels (32-pixel tile), channels not a multiple of 4
    (2, 8, 8, 128, 64, 3, 1, 1, 8, 4, 0, True),       # folded channel tile, packed 4-bit output
    (2, 8, 8, 80, 34, 1, 2, 0, 8, 4, 0, True),        # the same with channel pairs that do not fill words
    (2, 10, 10, 64, 192, 3, 1, 1, 4, 8, 8, True),     # packed 4-bit operands, shifts below 32 (64-bit form)
    (1, 7, 7, 16, 24, 3, 1, 1, 4, 4, 0, True),        # the smallest packed reduction step
    (37, 14, 14, 64, 64, 1, 1, 0, 8, 8, 0, True),     # more tiles than SMs: no split
    (1, 12, 300, 32, 8, 1, 1, 0, 8, 32, 0, False),    # wide rows, eight channels
]


@pytest.mark.parametrize("signed", [False, True])
@pytest.mark.parametrize("cfg", CASES)
def test_small_conv_kernel(cfg, signed):
    """Edges of the pixel, channel and reduction tiles, every split of the reduction, every operand and output type."""
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from oracle import hqref
    from paper_2011_10680_b200 import binding, build
    build.build()
    n, h, w, cin, cout, k, stride, pad, bits, out_bits, res_bits, relu = cfg
    case = inputs.conv_case(500, n, h, w, cin, cout, k, stride, pad, bits=bits, out_bits=out_bits, residual=res_bits > 0,
                            res_bits=res_bits or 8, relu=relu, in_signed=signed, c_range=(39, 44))
    hq = binding.Handle(0)
    try:
        hq.set_conv_path(4)
        dev = binding.upload_case(case)
        for _ in range(2):                                  # the second call starts while the first one ends
            st, out = hq.conv_case(case, dev)
            assert st == binding.HQ_OK, binding.status_string(st)
        hq.sync()
        ref = hqref.conv_case(case)
        got = out.cpu().numpy().view(ref.dtype).reshape(ref.shape)
        assert np.array_equal(got, ref), (int((got != ref).sum()), ref.size)
    finally:
        hq.close()


@pytest.mark.parametrize("shifts", ["table", "residual_below_32", "main_below_32", "every"])
def test_fused_int32_stream_add(shifts):
    """Graph replay runs the INT32 add and the next block's requantization behind the block's last convolution; with layer
    taps every layer runs alone.  Both against the oracle on a reduced table, with shifts that select each arithmetic form."""
    from paper_2011_10680_b200 import binding, build
    from test_gpu_parity import run_network_and_compare
    build.build()
    t = inputs.resnet_table(50, seed=8, image_hw=64, classes=24, width=32, int32_stream=True)
    g = inputs.rng(77, len(shifts))
    pick = lambda c, lo, hi: g.integers(lo, hi, size=c, dtype=np.int64).astype(np.int32)
    for l in t["layers"]:
        if shifts == "table" or l["op"] not in ("add", "requant"):
            continue
        c = l["cout"]
        if l["op"] == "add":
            l["c"] = pick(c, *{"residual_below_32": (33, 36), "main_below_32": (28, 34), "every": (30, 60)}[shifts])
            l["rc"] = pick(c, *{"residual_below_32": (29, 34), "main_below_32": (31, 34), "every": (30, 60)}[shifts])
        else:
            l["c"] = pick(c, *((40, 48) if shifts != "every" else (30, 50)))
    hq = binding.Handle(0)
    try:
        run_network_and_compare(hq, t, batch=3, seed=61)
    finally:
        hq.close()


def test_fused_int32_stream_add_large_tiles():
    """The same with 256-pixel tiles, folded channel tiles and several tiles per CTA (layers of 40 thousand pixels): the
    fused run against the layer-by-layer run, whose kernels other tests compare with the oracle."""
    from paper_2011_10680_b200 import binding, build
    build.build()
    t = inputs.resnet_table(50, seed=9, image_hw=96, classes=24, int32_stream=True)
    hq = binding.Handle(0)
    net = binding.Network(hq, t, 73)
    try:
        images = binding.to_device(inputs.random_images(5, 73, 96))
        single, fused = (binding.alloc_out(*net.logits_shape, 32, 1) for _ in range(2))
        assert net.run(images, single, net.alloc_taps()) == binding.HQ_OK
        hq.sync()
        with torch.cuda.stream(torch.cuda.Stream()):
            assert net.run(images, fused, None) == binding.HQ_OK
            hq.sync()
        net.check_guards()
        assert int((single != single[0]).sum()) > 0 and torch.equal(single, fused)
    finally:
        net.close()
        hq.close()


@pytest.mark.parametrize("path", [2, 4])
@pytest.mark.parametrize("cfg", [
    # n, h, w, cin, cout, k, stride, pad, bits, residual
    (9, 20, 20, 48, 64, 5, 1, 2, 8, False),      # one 64-byte block per tap, 16 bytes of it past the channels
    (9, 20, 20, 96, 96, 3, 1, 1, 8, False),      # 96 of 128
    (5, 20, 20, 144, 192, 3, 2, 1, 8, False),    # a full block and 16 of 128
    (9, 20, 20, 192, 256, 1, 1, 0, 8, True),     # tiled rows, residual
    (12, 30, 30, 16, 128, 3, 1, 1, 8, False),    # half a 32-byte block
    (4, 20, 20, 288, 256, 3, 1, 1, 8, False),    # long reduction: two full blocks and 32 of 128
    (41, 31, 31, 288, 256, 3, 1, 1, 8, False),   # the same with two tiles per SM: the two-CTA shape, a ragged last tile
    (9, 20, 20, 48, 64, 5, 1, 2, 4, False),      # widened 4-bit operands
])
def test_conv_channels_that_do_not_fill_a_block(cfg, path):
    """K blocks that reach past the channels of a tap, in both tensor-core kernels."""
    from oracle import hqref
    from paper_2011_10680_b200 import binding, build
    build.build()
    n, h, w, cin, cout, k, stride, pad, bits, residual = cfg
    case = inputs.conv_case(600, n, h, w, cin, cout, k, stride, pad, bits=bits, residual=residual, c_range=(38, 44))
    ref = hqref.conv_case(case)
    hq = binding.Handle(0)
    try:
        for p in ((2, 3) if path == 2 else (4,)):
            hq.set_conv_path(p)
            st, out = hq.conv_case(case)
            assert st == binding.HQ_OK, binding.status_string(st)
            hq.sync()
            assert np.array_equal(out.cpu().numpy().view(ref.dtype).reshape(ref.shape), ref)
    finally:
        hq.close()


@pytest.mark.parametrize("signed,shift", [(False, None), (True, None), (True, 28), (False, 31)])
def test_fused_pooling_branch(signed, shift):
    """Graph replay rescales the window sums of a pooling branch straight into the concatenation: unsigned and signed module
    inputs, shifts on both sides of 32, a branch at either end; ragged last strip (9 rows).  Oracle through the layer taps."""
    from paper_2011_10680_b200 import binding, build
    from test_gpu_parity import run_network_and_compare
    build.build()
    bd = inputs._Builder(31)
    bd.scale[-1], bd.shape[-1], bd.bits[-1] = 2.0 ** -4, (20, 20, 3), 8
    x = bd.conv(-1, 48, 3, 2, 0, 8, relu=not signed, out_bits=8, out_signed=signed)
    for last in (True, False):
        m = bd.conv(x, 36, 1, 1, 0, 8, relu=True, out_bits=8)
        p = bd.sumpool(x, 3, 1, 1)
        x = bd.concat([m, p] if last else [p, m])
        if shift:
            k = bd.layers[x]["ins"].index(p)
            bd.layers[x]["cs"][k][::3] = shift
    x = bd.avgpool(x)
    bd.conv(x, 16, 1, 1, 0, 8, relu=False, out_bits=32, op="linear")
    t = dict(layers=bd.layers, image_hw=20, classes=16, depth=0, conv_bits=[8], shapes=[bd.shape[i] for i in range(len(bd.layers))],
             bits=[bd.bits[i] for i in range(len(bd.layers))])
    hq = binding.Handle(0)
    try:
        run_network_and_compare(hq, t, batch=3, seed=6)
    finally:
        hq.close()


@pytest.mark.parametrize("hw,batch,signed", [(56, 11, False), (50, 13, True), (26, 41, False)])
def test_conv_over_pixel_pairs(hw, batch, signed):
    """3x3 layers of 64 channels in the pixel-pair form of a network: full and ragged tiles, both pitches, signed outputs."""
    from paper_2011_10680_b200 import binding, build
    from test_gpu_parity import run_network_and_compare
    build.build()
    bd = inputs._Builder(hw)
    bd.scale[-1], bd.shape[-1], bd.bits[-1] = 2.0 ** -4, (2 * hw, 2 * hw, 3), 8
    x = bd.conv(-1, 64, 3, 2, 1, 8, relu=True, out_bits=8)
    x = bd.conv(x, 64, 3, 1, 1, 8, relu=not signed, out_bits=8, out_signed=signed)
    x = bd.conv(x, 64, 3, 1, 1, 8, relu=True, out_bits=8)
    x = bd.avgpool(x)
    bd.conv(x, 16, 1, 1, 0, 8, relu=False, out_bits=32, op="linear")
    t = dict(layers=bd.layers, image_hw=2 * hw, classes=16, depth=0, conv_bits=[8], shapes=[bd.shape[i] for i in range(len(bd.layers))],
             bits=[bd.bits[i] for i in range(len(bd.layers))])
    hq = binding.Handle(0)
    try:
        run_network_and_compare(hq, t, batch=batch, seed=6)
    finally:
        hq.close()


FRAGMENT_CASES = [
    # n, h, w, cin, cout, k, stride, residual, residual signed, relu, c range, rc range,
    #   plan on 148 SMs: K blocks, stages, MMA issue (whole tiles in turn / K blocks dealt in turn), residual or output tiles, weights resident
    (258, 28, 27, 32, 144, 1, 1, True, False, True, (39, 44), (28, 34), (1, 8, "tiles", 8, 1)),     # blocks of 32 bytes; second channel tile of 16; ragged last pixel tile
    (258, 28, 27, 64, 256, 1, 1, True, True, False, (39, 44), (28, 34), (1, 8, "tiles", 8, 1)),     # signed residual and output
    (258, 28, 27, 96, 160, 1, 1, True, False, True, (39, 44), (28, 34), (1, 4, "tiles", 8, 1)),     # the last K block reaches past the channels
    (258, 28, 27, 128, 256, 1, 1, True, False, True, (28, 31), (28, 34), (1, 4, "tiles", 8, 1)),    # shifts below 32: pre-shift form
    (258, 28, 27, 64, 256, 1, 1, True, False, True, (14, 40), (28, 34), (1, 8, "tiles", 8, 1)),     # some shifts too small for it: funnel-shift form
    (258, 28, 27, 64, 256, 1, 1, True, True, True, (39, 44), (4, 34), (1, 8, "tiles", 8, 1)),       # residual shifts below 9: 64-bit form
    (258, 28, 27, 256, 256, 1, 1, True, False, True, (39, 44), (28, 34), (2, 4, "blocks", 8, 1)),   # each issuer keeps one block of every tile
    (258, 28, 27, 160, 256, 1, 1, True, False, True, (39, 44), (28, 34), (2, 4, "blocks", 8, 1)),   # the same with a partial last block
    (258, 28, 27, 320, 256, 1, 1, True, False, True, (39, 44), (28, 34), (3, 6, "blocks", 4, 1)),   # three blocks: the issuers swap roles from tile to tile
    (258, 28, 27, 64, 256, 3, 1, True, False, True, (39, 44), (28, 34), (9, 8, "blocks", 4, 1)),    # nine blocks, rows gathered in im2col mode
    (258, 28, 27, 32, 256, 3, 1, True, True, True, (39, 44), (28, 34), (9, 8, "blocks", 4, 1)),     # nine blocks of 32 bytes
    (130, 28, 27, 512, 512, 1, 1, True, False, True, (40, 45), (28, 34), (4, 6, "blocks", 4, 1)),   # four blocks
    (130, 28, 27, 640, 512, 1, 1, True, False, True, (40, 45), (28, 34), (5, 4, "blocks", 4, 0)),   # five blocks, weights in the stages
    (258, 28, 27, 64, 256, 1, 1, False, False, True, (39, 44), None, (1, 8, "tiles", 4, 1)),        # no residual
    (258, 28, 27, 64, 176, 1, 1, False, False, False, (26, 44), None, (1, 8, "tiles", 4, 1)),       # the same, signed, ragged channels, small shifts
    (980, 28, 27, 256, 256, 1, 2, False, False, True, (39, 44), None, (2, 8, "tiles", 4, 1)),       # the same, rows gathered in im2col mode
    (258, 28, 27, 384, 256, 1, 1, False, False, True, (39, 44), None, (3, 8, "blocks", 2, 1)),      # three blocks without a residual, two output tiles
]


@pytest.mark.parametrize("rev", [0, 1])
@pytest.mark.parametrize("cfg", FRAGMENT_CASES)
def test_fragment_epilogue_shape(cfg, rev):
    """The launch shape with four accumulators and two groups of epilogue warps: every number of K blocks per tile, every form of
    the arithmetic, ragged channel and pixel tiles, both tile orders, and enough tiles that every ring of buffers comes round twice
    (two distinct images, repeated: the output must repeat with them).  Integers: equal to the oracle.  That each case takes
    the plan it names is checked without a GPU (test_conv_plan.py)."""
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from oracle import hqref
    from paper_2011_10680_b200 import binding, build
    build.build()
    n, h, w, cin, cout, k, stride, residual, res_signed, relu, c_range, rc_range, _ = cfg
    case = inputs.conv_case(700, 2, h, w, cin, cout, k, stride, k // 2, residual=residual, relu=relu, c_range=c_range)
    if residual:
        g = inputs.rng(701, cin, cout, k)
        case["rc"] = g.integers(rc_range[0], rc_range[1] + 1, size=cout, dtype=np.int64).astype(np.int32)
        if res_signed:
            case["res"], case["res_signed"] = case["res"].view(np.int8), 1
    big = dict(case, n=n, x=np.tile(case["x"], (n // 2, 1, 1, 1)))
    if residual:
        big["res"] = np.tile(case["res"], (n // 2, 1, 1, 1))
    ref = hqref.conv_case(case)
    hq = binding.Handle(0)
    try:
        hq.set_tile_order(rev)
        dev = binding.upload_case(big)
        for _ in range(2):                                  # the second call starts while the first one ends
            st, out = hq.conv_case(big, dev)
            assert st == binding.HQ_OK, binding.status_string(st)
        hq.sync()
        got = out.cpu().numpy().view(ref.dtype).reshape(n // 2, *ref.shape)
        assert np.array_equal(got, np.broadcast_to(ref, got.shape)), (int((got != ref).sum()), got.size)
    finally:
        hq.close()
