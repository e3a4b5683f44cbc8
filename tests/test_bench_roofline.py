"""bench.py's roofline line: the DRAM bytes beside a kernel's time are that kernel's own."""
import argparse
import json
import os
import re

import bench
from paper_2605_05888_b200 import inputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def options(**kw):
    return argparse.Namespace(**{"tp_shards": 0, "ffn_kernel": 0, "ffn_split": 0, "overlap": 0, "ffn_hot_min_tiles": 0, "ffn_thin_tiles": 0, **kw})


def test_the_kernel_follows_the_plan_options():
    c3, c2, qwen = bench.WORKLOADS["c3"], bench.WORKLOADS["c2"], bench.WORKLOADS["c4"]
    assert bench.expert_kernel(options(), c3) == bench.expert_kernel(options(), c2) == "ffn_pair_kernel"
    assert bench.expert_kernel(options(overlap=1), c3) == bench.expert_kernel(options(ffn_thin_tiles=-1), c3) == "ffn_tc_kernel"
    assert bench.expert_kernel(options(), qwen) == "ffn_tc_kernel"
    assert bench.expert_kernel(options(), qwen.with_(T=5)) == "few-token kernels"
    assert bench.expert_kernel(options(ffn_split=2), qwen.with_(T=5)) == "ffn_tc_kernel"


def test_traffic_is_null_for_a_kernel_without_a_capture():
    with open(os.path.join(ROOT, "profiles", "ncu_dram_traffic.json")) as f:
        kept = {k: v for k, v in json.load(f).items() if k != "what"}
    sources = "".join(open(os.path.join(ROOT, "paper_2605_05888_b200", "csrc", n)).read()
                      for n in os.listdir(os.path.join(ROOT, "paper_2605_05888_b200", "csrc")) if n.endswith(".cu"))
    for workload, kernels in kept.items():
        for kernel, entry in kernels.items():
            assert re.search(rf"^{kernel}\(", sources, re.M), f"no kernel of that name: {kernel}"
            assert os.path.exists(os.path.join(ROOT, re.match(r"[\w/]+\.md", entry["source"]).group(0)))
            assert bench.ncu_traffic_bytes(workload, kernel) == entry["bytes"]
        assert bench.ncu_traffic_bytes(workload, "few-token kernels") is None
    name = bench.WORKLOADS["c3"].name
    assert bench.ncu_traffic_bytes(name, "ffn_pair_kernel") != bench.ncu_traffic_bytes(name, "ffn_tc_kernel")
