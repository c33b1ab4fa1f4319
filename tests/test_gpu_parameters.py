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
