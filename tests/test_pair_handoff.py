"""What one CTA of decode_pair writes and the other's issuer reads is released to the
cluster and acquired from it: an arrival and a probe have the scope of their own CTA by
default, which leaves the mark of a raise invisible to the issuer however long ago its
warp arrived (the model in test_pair_protocol_model.py shows PV then reading weights that
are being rewritten)."""
import os
import re

import pytest

from paper_2609_36760_gb300 import build


def _source(name):
    text = open(os.path.join(build.CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


PAIR = _source("decode_pair.cu")


@pytest.mark.parametrize("helper,op", [
    ("mbar_arrive_cluster", "mbarrier.arrive.release.cluster.shared::cluster.b64"),
    ("mbar_test_cluster", "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64"),
])
def test_cluster_scope_helpers(helper, op):
    body = re.search(helper + r"\([^)]*\)\s*\{(.*?)\n\}", _source("ptx.cuh"), re.S)
    assert body and op in body.group(1)


def test_the_arrival_behind_a_mark_is_a_cluster_release():
    assert re.search(r"arrive_leader_cluster\([^)]*\)\s*\{\s*mbar_arrive_cluster\(", PAIR)
    mark = PAIR.index("st_cluster_u32(cluster_map(smem_u32(&ctl.raised")
    after = re.search(r"arrive_leader(_cluster)?\(lane, (\w+)", PAIR[mark:])
    assert after.groups() == ("_cluster", "pfull")
    # and the rewritten weights'
    assert re.findall(r"arrive_leader(_cluster)?\(lane, pfixed\)", PAIR) == ["_cluster"]


@pytest.mark.parametrize("bar", ["k_full", "v_full", "p_full", "p_fixed", "s_free", "o_free", "q_peer"])
def test_the_issuer_acquires_from_the_cluster(bar):
    issuer = PAIR[PAIR.index("void pair_mma("):PAIR.index("void pair_query(")]
    assert re.findall(r"(mbar_\w+)\(&ctl\." + bar, issuer) == ["mbar_test_cluster"]
