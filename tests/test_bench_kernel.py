"""The bench line names the main kernel that its workload runs, and takes traffic figures
of that kernel only."""
import json
import os
import sys
import types

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import paper_2609_36760_gb300 as Q  # noqa: E402
from workloads import synthetic as W  # noqa: E402


@pytest.mark.parametrize("name,bf16,kernel", [
    ("dsv3_b64_h128_l4096_int4", False, "decode_pair"), ("dsv3_b64_h128_l4096_int4", True, "decode_pair"),
    ("int2_b32_h128_l32768", False, "decode_pair"), ("serve_b128_h16_mix", False, "decode_main"),
    ("tiny_b1_h16_l256_int4", False, "decode_main"),
])
def test_kernel_of_a_workload(name, bf16, kernel):
    import bench
    st = object.__new__(bench.Workspace)
    st.w, st.bf16, st.c4r4, st.protect, st.q_tokens = W.WORKLOADS[name], bf16, False, False, 1
    st.table, _ = W.block_table(st.w)
    st.Q = types.SimpleNamespace(debug_decode_route=Q.debug_decode_route, num_sms=lambda: 152)
    assert st.kernel() == kernel and kernel in bench.KERNELS[st.kernel()]


def test_traffic_is_the_kernel_s_own(tmp_path, monkeypatch):
    import bench
    os.makedirs(tmp_path / "profiles")
    rec = {"kernel": "decode_pair", "workload": "x", "dram_bytes_per_launch": 5, "source": "s"}
    (tmp_path / "profiles" / "decode_traffic.json").write_text(
        json.dumps({"decode_sources_sha256": "h", "records": [rec]}))
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.profile_traffic("h", "decode_pair", "x") == rec
    assert bench.profile_traffic("h", "decode_main", "x") is None
    assert bench.profile_traffic("other", "decode_pair", "x") is None
