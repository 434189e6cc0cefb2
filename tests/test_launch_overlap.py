"""The overlap of a cache writer and the decode behind it. The writers let the decode's
first kernel (prep) start beside them, so prep must not write before it has waited for
the writer: its workspace may be memory that the writer still reads (in stream order a
program may free the latents behind the append and allocate the workspace in their
place)."""
import os
import re

import numpy as np
import pytest
import torch

import paper_2609_36760_gb300 as Q
from paper_2609_36760_gb300 import build

SRC = os.path.join(build.CSRC, "decode.cu")


def _body(text, head):
    """The braces' content of the function whose declaration contains `head`."""
    at = text.index("{", text.index(head))
    depth, i = 0, at
    while True:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
        if depth == 0:
            return re.sub(r"//[^\n]*", "", text[at:i])


@pytest.mark.parametrize("head,writes", [
    ("void query_piece(", r"reinterpret_cast<uint4\*>\(img"),
    ("prep_kernel(const Params p)", r"p\.(?:prefix_w|cta_info|cta_first|cta_t0)\[[^\]]*\]\s*=[^=]"),
    ("prep_kernel(const Params p)", r"\bpf\[[^\]]*\]\s*=[^=]"),  # the workspace's prefix where it is not on chip
])
def test_prep_waits_before_its_first_write(head, writes):
    body = _body(open(SRC).read(), head)
    first = re.search(writes, body)
    assert first is not None
    assert "griddep_wait();" in body[:first.start()]


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["int4", "bf16"])
@pytest.mark.parametrize("batch,heads", [(8, 128), (8, 16), (4200, 16)])  # 4,200 units: the prefix not on chip
def test_workspace_in_the_memory_of_the_written_latents(kind, batch, heads):
    # many more tokens than the writer has in flight at once, the workspace over the last ones
    per = max(10, 40000 // batch)
    n = batch * per
    cols = (per + 63) // 64
    g = torch.Generator(device="cuda").manual_seed(batch + heads)
    lat = torch.randn(n, 512, generator=g, device="cuda").bfloat16()
    kpe = torch.randn(n, 64, generator=g, device="cuda").bfloat16()
    sid = torch.arange(n, dtype=torch.int32, device="cuda") // per
    pos = torch.arange(n, dtype=torch.int32, device="cuda") % per
    table = torch.arange(batch * cols, dtype=torch.int32, device="cuda").view(batch, cols)
    lens = torch.full((batch,), per, dtype=torch.int32, device="cuda")
    ql = (torch.randn(batch, heads, 512, generator=g, device="cuda") / 22.6).bfloat16()
    qp = (torch.randn(batch, heads, 64, generator=g, device="cuda") / 8.0).bfloat16()
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    bb = Q.bf16_block_bytes() if kind == "bf16" else Q.block_bytes(4)
    need = (Q.workspace_for(batch, heads).nbytes + 255) // 256 * 256
    size = max(need, lat.nbytes)

    def run(shared):
        pool = torch.zeros((batch * cols, bb), dtype=torch.uint8, device="cuda")
        out = torch.empty((batch, heads, 512), dtype=torch.float32, device="cuda")
        lse = torch.empty((batch, heads), dtype=torch.float32, device="cuda")
        room = torch.zeros(size, dtype=torch.uint8, device="cuda")
        src = room[size - lat.nbytes:].view(torch.bfloat16).view(n, 512)
        src.copy_(lat)
        ws = room[size - need:] if shared else torch.empty(need, dtype=torch.uint8, device="cuda")
        if kind == "bf16":
            Q.bf16_append(pool, src, kpe, sid, pos, table, err)
            Q.mla_decode_bf16cache(pool, ql, qp, table, lens, 0.07, out, lse, ws, err)
        else:
            Q.quant_append(pool, 4, src, kpe, sid, pos, table, err)
            Q.mla_decode(pool, 4, ql, qp, table, lens, 0.07, out, lse, ws, err)
        torch.cuda.synchronize()
        return pool.cpu().numpy(), out.cpu().numpy(), lse.cpu().numpy()

    want, got = run(False), run(True)
    assert Q.read_dev_err(err) == 0
    for a, b in zip(want, got):
        assert np.array_equal(a, b)
