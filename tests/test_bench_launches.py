"""The benchmark's count of this library's launches per pp_layer call, against
the launch lists of the timed regions in profiles/ (kernel rows, launches)."""
import os
import re

import bench
from paper_2605_28283_gb300 import workloads as wl

LISTS = [("llama2_7b_decode", 1, "decode_layer_llama2_7b_b1_p0.7_launches.md", 512),
         ("gpt2m_gelu_bf16", 4, "decode_layer_gpt2m_b4_p0.7_launches.md", 384),
         ("llama3_8b_batched", 64, "grouped_llama3_8b_b64_p0.7_launches.md", 128),
         ("llama2_13b_prefill", 8192, "prefill_llama2_13b_t8192_launches.md", 2)]


def test_launches_per_call_match_the_launch_lists():
    for name, B, path, calls in LISTS:
        text = open(os.path.join(os.path.dirname(bench.__file__), "profiles", path)).read()
        rows = re.findall(r"^\| `pp::[^|]*\| (\d+) \|", text, re.M)
        assert sum(map(int, rows)) == calls * bench.kernels_per_call(wl.WORKLOADS[name], B), path


def test_launches_per_call_at_the_edges():
    bf16, f32 = wl.WORKLOADS["llama3_8b_batched"], wl.WORKLOADS["tiny_relu_f32"]
    assert [bench.kernels_per_call(bf16, B) for B in (1, 4, 5, 256, 257)] == [1, 1, 1, 1, 5]
    assert [bench.kernels_per_call(f32, B) for B in (1, 8, 9, 2000)] == [1, 1, 3, 3]
