"""That the tests which compare decode_pair with decode_main run both: the narrow table of
some of tests/test_gpu_pair.py's cases lies close to the pair's threshold, and the BF16
case of its raises is beyond it, so that both of its runs take the pair."""
import numpy as np
import pytest
import torch

import paper_2609_36760_gb300 as Q
from harness import TAU, Case, rel_l2
from test_gpu_pair import RAGGED, SPLIT
from workloads import synthetic as W

WIDE = 4096


def _cols(lengths):
    return (max(lengths) + 63) // 64


@pytest.mark.parametrize("lengths", [RAGGED, SPLIT])
@pytest.mark.parametrize("kind,protect", [(4, False), (4, True), (2, False), (2, True), ("c4r4", False),
                                          ("c4r4", True), ("bf16", False)])
def test_pair_comparisons_run_both_kernels(kind, protect, lengths):
    for heads in (65, 100, 128):
        got = [Q.debug_decode_route(kind, len(lengths), heads, c, protect=protect) for c in (_cols(lengths), WIDE)]
        assert got == ["decode_main", "decode_pair"]
    for t, heads in ((2, 64), (2, 128), (4, 32), (3, 128)):
        if kind != 4 or not protect:
            continue
        got = [Q.debug_decode_route(4, 6, heads, c, q_tokens=t, protect=True) for c in (_cols([700]), WIDE)]
        assert got == ["decode_main", "decode_pair"]


@pytest.mark.gpu
@pytest.mark.parametrize("kind,protect", [("bf16", False), ("int4", True)])
def test_raises_inside_a_range_on_both_kernels(kind, protect):
    # As test_pair_raises_inside_a_range, for caches whose narrow table is already wide
    # enough for the pair: decode_main's side by a bound of one token. Same tolerances.
    lengths = (9000, 8000, 9500, 7000)
    w = W.small_workload("r", batch=4, heads=128, lengths=lengths, c_bits=4, seed=72)
    c = Case(w, bf16_cache=kind == "bf16", protect=protect)
    ql, qp = W.queries(w, 0)
    for b in range(w.batch):
        lat, kp = c.tokens(b)
        lat = lat.double() * 0.2
        for i, at in enumerate(range(170 + 17 * b, lat.shape[0], 450)):
            q = ql.double()[b, 5 * i % 128]
            lat[at] = q / q.norm() * lat[at].norm() * (1.2, 1.8, 3.0)[i % 3]
        c._tok[b] = (lat.to(torch.bfloat16), kp)
    c.prefill_all()
    ql = (ql.double() * 12.0).to(torch.bfloat16).cuda()
    sl = torch.tensor(lengths, dtype=torch.int32, device="cuda")
    ws = Q.workspace_for(4, 128)
    got = {}
    for max_len in (0, 1):
        out = torch.full((4, 128, 512), float("nan"), device="cuda")
        lse = torch.full((4, 128), float("nan"), device="cuda")
        code = "bf16" if kind == "bf16" else 4
        route = Q.debug_decode_route(code, 4, 128, c.table_d.shape[1], protect=protect, max_len=max_len,
                                     sms=Q.num_sms())
        Q.mla_decode_ex(c.pool, code, ql, qp.cuda(), c.table_d, sl, TAU, out, lse, ws, c.dev_err, prot=c.prot,
                        max_len=max_len)
        torch.cuda.synchronize()
        got[route] = out.cpu().numpy(), lse.cpu().numpy()
    assert c.dev_error() == 0 and set(got) == {"decode_main", "decode_pair"}
    (out_n, lse_n), (out_w, lse_w) = got["decode_main"], got["decode_pair"]
    for b in range(4):
        assert rel_l2(out_w[b], out_n[b]) <= 2.0 ** -11, b
        assert np.max(np.abs(lse_w[b] - lse_n[b])) <= 2.0 ** -11 * max(1.0, np.max(np.abs(lse_n[b])))
        ref, rlse = c.oracle_decode(b, c.prefill[b], 0, fp16_tiles=True, queries=(ql.cpu(), qp))
        assert rel_l2(out_w[b], ref) <= 1e-3
        assert np.max(np.abs(lse_w[b] - rlse)) <= 1e-3 * max(1.0, np.abs(rlse).max())
