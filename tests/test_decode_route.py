"""Which main kernel a decode runs on: by the table's width, or by the caller's bound of
the lengths. Short sequences in a table for 128K tokens are up to 14% slower on the pair
than on decode_main, which the table's width alone cannot tell."""
import numpy as np
import pytest
import torch

import paper_2609_36760_gb300 as Q
from harness import TAU, Case
from workloads import synthetic as W

WIDE = 4096


def _cols(lengths):
    return (max(lengths) + 63) // 64


@pytest.mark.parametrize("kind,batch,heads,length", [
    (4, 16, 128, 2000), (2, 16, 128, 2000), (2, 64, 128, 1000), ("c4r4", 16, 128, 1000), (4, 64, 128, 256),
    ("bf16", 1, 128, 128),
])
def test_a_bound_of_the_lengths_undoes_a_wide_table(kind, batch, heads, length):
    cut = Q.debug_decode_route(kind, batch, heads, _cols([length]))
    assert cut == "decode_main"
    assert Q.debug_decode_route(kind, batch, heads, 2048) == "decode_pair"
    assert Q.debug_decode_route(kind, batch, heads, 2048, max_len=length) == cut
    # a bound beyond the table is the table's; none, or less than one, is none
    for none in (0, -5, 1 << 30):
        assert Q.debug_decode_route(kind, batch, heads, 2048, max_len=none) == "decode_pair"
        assert Q.debug_decode_route(kind, batch, heads, _cols([length]), max_len=none) == cut


def test_rows_without_a_pair():
    for heads in (16, 64):
        assert Q.debug_decode_route(4, 64, heads, WIDE) == "decode_main"
    assert Q.debug_decode_route(4, 64, 64, WIDE, q_tokens=3) == "decode_main"  # three groups
    assert Q.debug_decode_route(4, 64, 64, WIDE, q_tokens=2) == "decode_pair"
    with pytest.raises(ValueError):
        Q.debug_decode_route(4, 0, 64, WIDE)


@pytest.mark.gpu
def test_a_bound_gives_the_cut_table_s_result():
    lengths = (300, 1, 1000, 640)
    w = W.small_workload("h", batch=4, heads=128, lengths=lengths, seed=5)
    c = Case(w)
    c.prefill_all()
    want = c.decode(0, lens=list(lengths))
    wide = torch.full((4, WIDE), -1, dtype=torch.int32, device="cuda")
    wide[:, :c.table_d.shape[1]] = c.table_d
    ql, qp = W.queries(w, 0)
    sl = torch.tensor(lengths, dtype=torch.int32, device="cuda")
    out = torch.full((4, 128, 512), float("nan"), device="cuda")
    lse = torch.full((4, 128), float("nan"), device="cuda")
    ws = Q.workspace_for(4, 128)
    Q.mla_decode_ex(c.pool, 4, ql.cuda(), qp.cuda(), wide, sl, TAU, out, lse, ws, c.dev_err, max_len=1000)
    assert c.dev_error() == 0
    # the same kernel over the same plan
    assert np.array_equal(out.cpu().numpy(), want[0]) and np.array_equal(lse.cpu().numpy(), want[1])
    # a bound that is too small chooses badly and changes no result
    out.fill_(float("nan"))
    Q.mla_decode_ex(c.pool, 4, ql.cuda(), qp.cuda(), wide, sl, TAU, out, lse, ws, c.dev_err, max_len=1)
    assert c.dev_error() == 0 and np.array_equal(out.cpu().numpy(), want[0])
