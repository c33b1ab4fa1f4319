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
