"""Launch plans of the persistent convolution kernel: host arithmetic, checked without a GPU over the sizes the kernel takes."""
from __future__ import annotations

import itertools
import os
import re

import pytest

from paper_2011_10680_b200 import binding, build

SMS = 148
PIXELS = (52, 28, 27)                        # 39312 pixels: 256-pixel tiles of two channel tiles fill the SMs twice


@pytest.fixture(scope="module", autouse=True)
def library():
    build.build()


def all_plans():
    """Every K-block size and count, one to five channel tiles, with and without a residual, whole and ragged channels."""
    small, large = (2, 14, 14), PIXELS
    for cin, (k, stride), cout, res, out_bits, (n, h, w) in itertools.product(
            [*range(16, 529, 16), 640, 768, 896, 1008, 1024, 2048], [(1, 1), (1, 2), (3, 1), (3, 2)], [64, 128, 144, 256, 512, 640],
            [0, 8, 32], [8, 4, 32], [small, large]):
        if res and out_bits != 8:
            continue
        plan = binding.conv2d_plan(n * stride * stride, h, w, cin, cout, k, stride, k // 2, out_bits, res, SMS)
        if plan is not None:
            yield (n, h, w, cin, cout, k, stride, res, out_bits), plan


def test_a_stage_belongs_to_one_issuer():
    """An issuer waits for the fill of a stage by its parity, so it has to have seen the fill before: whatever a stage
    holds, from one end of the launch to the other, goes to the same issuer.  Otherwise a copy that is overtaken by the
    next tiles lets the other issuer multiply what was there before."""
    seen = set()
    for layer, plan in all_plans():
        stages, issuers, blocks = plan["stages"], plan["issuers"], plan["k_blocks"]
        if issuers < 2 or not stages:
            continue
        seen.add((plan["shape"], stages, issuers, blocks, plan["alternate_tiles"]))
    assert {("frag", 1), ("frag", 0), ("solo", 0)} <= {(s[0], s[4]) for s in seen}
    for shape, stages, issuers, blocks, alternate in seen:
        owner = {}
        for block in range(4 * stages * issuers * blocks):
            issuer = (block // blocks if alternate else block) % issuers
            assert owner.setdefault(block % stages, issuer) == issuer, (shape, stages, issuers, blocks, alternate)


def test_fragment_shape_has_stages_for_both_issuers():
    """The residual tiles must not take the room of the operand stages: one issuer alone sets the tile rate of this shape."""
    plans = [(layer, plan) for layer, plan in all_plans() if plan["shape"] == "frag"]
    assert {plan["weights_resident"] for _, plan in plans} == {0, 1}
    for layer, plan in plans:
        assert plan["stages"] >= 4 and plan["issuers"] == 2, (layer, plan)


def test_cases_of_the_fragment_shape_take_the_plans_they_name():
    from test_gpu_small_conv import FRAGMENT_CASES
    dealt = set()
    for n, h, w, cin, cout, k, stride, residual, _, _, _, _, (blocks, stages, issue, tiles, resident) in FRAGMENT_CASES:
        plan = binding.conv2d_plan(n, h, w, cin, cout, k, stride, k // 2, 8, 8 if residual else 0, SMS)
        got = (plan["shape"], plan["issuers"], plan["k_blocks"], plan["stages"], "tiles" if plan["alternate_tiles"] else "blocks",
               plan["residual_tiles"], plan["weights_resident"])
        assert got == ("frag", 2, blocks, stages, issue, tiles, resident), (cin, cout, k, got)
        if issue == "blocks":
            dealt.add(blocks % 2)
        pixels, channel_tiles = n * ((h - 1) // stride + 1) * ((w - 1) // stride + 1), (cout + 127) // 128
        assert pixels % 128 and pixels // 128 // (SMS // channel_tiles) >= 20            # tiles per CTA: eight buffers come round twice
    assert dealt == {0, 1}


def test_plans_fit_the_sm():
    for layer, plan in all_plans():
        assert plan["shared_bytes"] <= 227 * 1024, (layer, plan)
        assert plan["stages"] >= 2 or plan["shape"] == "strip", (layer, plan)
        assert plan["issuers"] <= max(1, plan["stages"]) or plan["shape"] == "strip", (layer, plan)


def test_signals_between_tensor_core_threads_are_fenced():
    """What one thread's tensor-core operations did is ordered before another's only by a pair of fences around the barrier: every
    arrival that says "my MMA is issued" or "my loads are done" has its half directly ahead of it."""
    path = os.path.join(os.path.dirname(build.__file__), "csrc", "conv_tc.cu")
    code = re.sub(r"//[^\n]*", "", open(path).read())
    code = re.sub(r"\s+", " ", code)
    arrivals = list(re.finditer(r"mbar_arrive\(smem_u32\(&ctl\.(tstart|tempty)\[", code))
    assert {m.group(1) for m in arrivals} == {"tstart", "tempty"}
    for m in arrivals:
        assert re.search(r"tc_fence_before\(\); (__syncwarp\(\); )?(if \(lane == 0\) )?$", code[:m.start()]), code[m.start() - 80:m.end() + 10]
