"""The byte / operation model behind bench.py's roofline figures (host logic, no GPU): totals that the paper's
tables and simple counting fix."""
from __future__ import annotations

import bench
from paper_2011_10680_b200 import inputs


def test_resnet50_operation_count_matches_the_papers_bops_column():
    # Table 1b: ResNet-50 at W8A8 has 247 G BOPS = 64 x MACs, i.e. 3.86 G MACs per image (stride on the first 1x1)
    rows = bench.layer_work(bench.workload_table("resnet50_int8_b256"), 1)
    macs = sum(r["ops"] for r in rows) // 2
    assert abs(macs * 64 / 1e9 - 247) < 1.0


def test_bytes_count_every_operand_once_at_its_own_width():
    t = bench.workload_table("inception_modules_int4_b256")
    rows = bench.layer_work(t, 2)
    shapes, bits = t["shapes"], t["bits"]
    size = lambda i: 2 * shapes[i][0] * shapes[i][1] * shapes[i][2] * bits[i] // 8
    for r in rows:
        l = t["layers"][r["layer"]]
        if l["op"] == "concat":           # every branch (the INT32 pooling branch at four bytes a value) + the output
            assert r["bytes"] == sum(size(i) for i in l["ins"]) + size(r["layer"])
        elif l["op"] == "sumpool":        # 8-bit module input, INT32 sums
            assert r["bytes"] == size(l["in0"]) + size(r["layer"])
    # the INT32 residual stream moves several times the bytes of the fused 8-bit stream (Fig. 2 against the fused form)
    wide = sum(r["bytes"] for r in bench.layer_work(bench.workload_table("resnet50_int8_int32stream_b256"), 256))
    fused = sum(r["bytes"] for r in bench.layer_work(bench.workload_table("resnet50_int8_b256"), 256))
    assert 4.5 < wide / fused < 6.5


def test_layers_inside_another_launch_are_counted_there():
    t = bench.workload_table("resnet50_int8_int32stream_b256")
    layers, n = t["layers"], 2
    rows, single = bench.launch_work(t, n), bench.layer_work(t, n)
    assert sum(r["ops"] for r in rows) == sum(r["ops"] for r in single)
    values = lambda i: n * t["shapes"][i][0] * t["shapes"][i][1] * t["shapes"][i][2]
    adds = [i for i, l in enumerate(layers) if l["op"] == "add"]
    assert len(adds) == 16
    for i in adds:                                        # every residual add of the stream runs behind its block's last conv
        j = layers[i]["in0"]
        conv = layers[j]
        assert rows[j]["runs_in"] == i and rows[j]["bytes"] == 0 and rows[i]["conv"]
        quant = [m for m, l in enumerate(layers) if l["op"] == "requant" and l["in0"] == i]
        assert all(rows[m]["runs_in"] == i for m in quant)
        other = [m for m, l in enumerate(layers) if i in (l["in0"], l["in1"]) and m not in quant]
        out = values(i) * ((4 if other or not quant else 0) + sum(layers[m]["out_bits"] // 8 for m in quant))
        weights = conv["cout"] * (conv["kh"] * conv["kw"] * conv["cin"] + 13)
        res = values(i) * (4 if layers[layers[i]["in1"]]["out_bits"] == 32 else 1)
        assert rows[i]["bytes"] == values(conv["in0"]) + weights + res + out
    t = bench.workload_table("inception_modules_int4_b256")
    rows = bench.launch_work(t, n)
    pools = [i for i, l in enumerate(t["layers"]) if l["op"] == "sumpool"]
    assert pools and all(t["layers"][rows[i]["runs_in"]]["op"] == "concat" for i in pools)
    assert all(r["conv"] for r, l in zip(rows, t["layers"]) if l["op"] == "conv" and l["cin"] == 48)
    assert all(r["runs_in"] is None for r in bench.launch_work(bench.workload_table("resnet50_int8_b256"), n))
