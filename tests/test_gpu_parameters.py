"""When parameters are read, and which layers a network may run behind others: everything against the CPU oracle, bit-exact."""
from __future__ import annotations

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
