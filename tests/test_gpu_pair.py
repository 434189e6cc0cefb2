"""Decodes on CTA pairs (more than 64 query rows) against decode_main and the oracle.

The route is chosen by the block table's width, so the same inputs with a wide table
(unused columns -1) run on pairs and with a narrow one on decode_main. Both split the
sequences at other places but use the same softmax references, so their fp16 weights
are the same and the outputs differ by fp32 accumulation only: 2e-5 in the 2-norm is
about a hundred roundings of 2^-24 per element, and the wide run also has to meet the
oracle's bars. Where a reference has to be raised inside a sequence the weights are
rounded against other references, so only the oracle's bars hold."""
import numpy as np
import pytest
import torch

from harness import Case, rel_l2
from workloads import synthetic as W

pytestmark = pytest.mark.gpu

RAGGED = (1, 63, 64, 65, 127, 128, 129, 191, 193, 600, 0)
SPLIT = (2600, 1500, 1, 900, 64)  # more tiles than SMs: ranges begin inside units


def _widen(c, cols=4096):
    t = torch.full((c.w.batch, cols), -1, dtype=torch.int32)
    t[:, :c.table.shape[1]] = c.table
    c.table_d = t.to(c.dev)


def _case(kind, protect, heads, lengths, seed):
    bits = 2 if kind == "int2" else 4
    w = W.small_workload("p", batch=len(lengths), heads=heads, lengths=lengths, c_bits=bits, seed=seed,
                         latent_dist="t4_gain" if bits == 2 else "gauss_gain_outlier")
    c = Case(w, bf16_cache=kind == "bf16", protect=protect, c4r4=kind == "c4r4")
    c.prefill_all()
    return c


@pytest.mark.parametrize("lengths", [RAGGED, SPLIT])
@pytest.mark.parametrize("heads", [65, 100, 128])
@pytest.mark.parametrize("kind,protect", [("int4", False), ("int4", True), ("int2", False), ("int2", True),
                                          ("c4r4", False), ("c4r4", True), ("bf16", False)])
def test_pair_equals_single(kind, protect, heads, lengths):
    c = _case(kind, protect, heads, lengths, 300 + heads)
    out_n, lse_n = c.decode(0, lens=list(lengths))
    _widen(c)
    out_w, lse_w = c.decode(0, lens=list(lengths))
    assert c.dev_error() == 0
    for b, n in enumerate(lengths):
        if n == 0:
            assert np.all(out_w[b] == 0) and np.all(np.isneginf(lse_w[b]))
            continue
        assert rel_l2(out_w[b], out_n[b]) <= 2e-5, b
        assert np.max(np.abs(lse_w[b] - lse_n[b])) <= 2e-5 * max(1.0, np.max(np.abs(lse_n[b])))
        ref, rlse = c.oracle_decode(b, n, 0)
        assert rel_l2(out_w[b], ref) <= 1e-3
        assert np.max(np.abs(lse_w[b] - rlse)) <= 1e-3


@pytest.mark.parametrize("q_tokens,heads", [(2, 64), (2, 128), (4, 32), (3, 128)])
def test_pair_several_query_tokens(q_tokens, heads):
    lengths = (2, 64, 65, 129, 700, 3)
    c = _case("int4", True, heads, lengths, 41)
    out_n, lse_n = c.decode_multi(0, q_tokens, lens=list(lengths))
    _widen(c)
    out_w, lse_w = c.decode_multi(0, q_tokens, lens=list(lengths))
    assert c.dev_error() == 0
    assert rel_l2(out_w, out_n) <= 2e-5
    seen = np.isfinite(lse_n)
    assert np.array_equal(seen, np.isfinite(lse_w)) and np.all(out_w[~seen] == 0)
    assert np.max(np.abs(lse_w[seen] - lse_n[seen])) <= 2e-5 * np.max(np.abs(lse_n[seen]))


@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_pair_raised_and_falling_references(sign):
    # scores that grow (or fall) by far more than 2^8 along the sequences
    w = W.small_workload("r", batch=3, heads=128, lengths=(1500, 700, 2300), seed=71)
    c = Case(w)
    for b in range(w.batch):
        lat, kp = c.tokens(b)
        ramp = torch.linspace(0.2, 3.0, lat.shape[0], dtype=torch.float64)[:, None]
        c._tok[b] = ((lat.double() * (ramp if sign > 0 else ramp.flip(0))).to(torch.bfloat16), kp)
    c.prefill_all()
    _widen(c)
    ql, qp = W.queries(w, 0)
    ql = (ql.double() * 40.0).to(torch.bfloat16)
    out, lse = c.decode(0, queries=(ql, qp))
    assert c.dev_error() == 0 and np.isfinite(out).all()
    for b in range(w.batch):
        ref, rlse = c.oracle_decode(b, c.prefill[b], 0, fp16_tiles=True, queries=(ql, qp))
        assert np.max(np.abs(out[b] - ref)) <= 2e-3 * np.abs(ref).max()
        assert rel_l2(out[b], ref) <= 1e-3
        assert np.max(np.abs(lse[b] - rlse)) <= 1e-3 * max(1.0, np.abs(rlse).max())


def test_pair_bad_block_flags_error_and_spares_neighbours():
    c = _case("int4", False, 128, (300, 300), 9)
    _widen(c)
    good, _ = c.decode(0, lens=[300, 300])
    c.table_d[0, 2] = c.nblocks + 5
    out, lse = c.decode(0, lens=[300, 300])
    assert c.dev_error() == 1
    assert np.isfinite(out).all() and np.isfinite(lse).all()
    assert np.array_equal(out[1], good[1])


@pytest.mark.parametrize("kind", ["int4", "int2", "bf16"])
def test_pair_raises_inside_a_range(kind):
    # 564 tiles, several per range of the plan; single tokens that exceed the reference by
    # far more than 2^8 at places of either parity of block, some with most of the sum
    lengths = (9000, 8000, 9500, 7000)
    bits = 2 if kind == "int2" else 4
    w = W.small_workload("r", batch=4, heads=128, lengths=lengths, c_bits=bits, seed=72)
    c = Case(w, bf16_cache=kind == "bf16")
    ql, qp = W.queries(w, 0)
    for b in range(w.batch):
        lat, kp = c.tokens(b)
        lat = lat.double() * 0.2
        for i, at in enumerate(range(170 + 17 * b, lat.shape[0], 450)):
            q = ql.double()[b, 5 * i % 128]
            lat[at] = q / q.norm() * lat[at].norm() * (1.2, 1.8, 3.0)[i % 3]
        c._tok[b] = (lat.to(torch.bfloat16), kp)
    c.prefill_all()
    ql = (ql.double() * 12.0).to(torch.bfloat16)
    out_n, lse_n = c.decode(0, queries=(ql, qp))
    _widen(c)
    out_w, lse_w = c.decode(0, queries=(ql, qp))
    assert c.dev_error() == 0
    for b in range(w.batch):
        # the same references, but for the weights of the even blocks of tiles that an odd
        # block raised: 2^-11 of at most one block's share of the sum
        assert rel_l2(out_w[b], out_n[b]) <= 2.0 ** -11, b
        assert np.max(np.abs(lse_w[b] - lse_n[b])) <= 2.0 ** -11 * max(1.0, np.max(np.abs(lse_n[b])))
        ref, rlse = c.oracle_decode(b, c.prefill[b], 0, fp16_tiles=True, queries=(ql, qp))
        assert rel_l2(out_w[b], ref) <= 1e-3
        assert np.max(np.abs(lse_w[b] - rlse)) <= 1e-3 * max(1.0, np.abs(rlse).max())
