"""The cache writers' branches: one or four tokens per lane, 16-byte and 4-byte
loads, partial groups of tokens, and groups whose codes take IEEE divisions
(quotients above 2^14, infinite values, NaNs). Bytes are compared exactly."""
import numpy as np
import pytest
import torch

import paper_2609_36760_gb300 as Q
from oracle import layout as OL
from oracle import paper_format as OF

pytestmark = pytest.mark.gpu


def _inputs(n, seed):
    """Latents and keys whose groups span many scales and distances from zero."""
    g = torch.Generator().manual_seed(seed)
    x = torch.randn(n, 9, 64, generator=g, dtype=torch.float64)
    scale = 10.0 ** (torch.rand(n, 9, 1, generator=g, dtype=torch.float64) * 8 - 5)
    far = torch.rand(n, 9, 1, generator=g, dtype=torch.float64)
    x = x * scale + torch.where(far < 0.2, scale * 10.0 ** (far * 30), torch.zeros_like(far))
    x[torch.rand(n, 9, generator=g) < 0.1] = 0.75  # constant groups
    x = x.reshape(n, 576).to(torch.bfloat16)
    return x[:, :512].contiguous(), x[:, 512:].contiguous()


def _device(t, shift):
    """t on the GPU, starting `shift` bf16 elements into its allocation."""
    buf = torch.empty(t.numel() + shift, dtype=t.dtype, device="cuda")
    v = buf[shift:].view(t.shape)
    v.copy_(t)
    return v


def _append(kind, lat, kpe, shift):
    n = lat.shape[0]
    nblk = (n + 63) // 64
    table = torch.randperm(nblk, generator=torch.Generator().manual_seed(n)).int()[None, :]
    bb = {4: Q.block_bytes(4), 2: Q.block_bytes(2), "c4r4": Q.c4r4_page_bytes(), "bf16": Q.bf16_block_bytes()}[kind]
    pool = torch.full((nblk, bb), 0xAB, dtype=torch.uint8, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    sid = torch.zeros(n, dtype=torch.int32, device="cuda")
    pos = torch.arange(n, dtype=torch.int32, device="cuda")
    l, k, t = _device(lat, shift), _device(kpe, shift), table.cuda()
    if kind == "c4r4":
        Q.quant_append_c4r4(pool, l, k, sid, pos, t, err)
    elif kind == "bf16":
        Q.bf16_append(pool, l, k, sid, pos, t, err)
    else:
        Q.quant_append(pool, kind, l, k, sid, pos, t, err)
    torch.cuda.synchronize()
    assert Q.read_dev_err(err) == 0
    return pool.cpu().numpy(), table.numpy()


@pytest.mark.parametrize("shift", [0, 2])
@pytest.mark.parametrize("n", [1, 3, 4, 129, 8191, 8192, 8207])
@pytest.mark.parametrize("kind", [4, 2, "c4r4", "bf16"])
def test_bytes_of_every_path(kind, n, shift):
    lat, kpe = _inputs(n, 17 * n + 1)
    got, table = _append(kind, lat, kpe, shift)
    want = np.full_like(got, 0xAB)
    sid, pos = np.zeros(n, np.int64), np.arange(n)
    if kind == "c4r4":
        OF.write_tokens(want, lat.double().numpy(), kpe.double().numpy(), sid, pos, table)
    elif kind == "bf16":
        rows = torch.cat([lat, kpe], 1).view(torch.int16).numpy().view(np.uint8)
        want.reshape(-1, 64, 1152)[table[0][pos // 64], pos % 64] = rows
    else:
        OL.write_tokens(want, kind, lat.double().numpy(), kpe.double().numpy(), sid, pos, table)
    assert np.array_equal(got, want)


def _group(x, bits, kind):
    """One group by the header's formulas in fp32 with IEEE division; minimum and
    maximum ignore NaNs, a NaN code or zero point is 0."""
    f = np.float32
    m = f(2 ** bits - 1)
    with np.errstate(all="ignore"):
        lo, hi = np.fmin.reduce(x), np.fmax.reduce(x)
        s = f(np.fmax(f(hi - lo), f(1e-8)) / m)
        if kind == "own":
            s = f(np.float16(s))
            s = f(2.0 ** -24) if s == 0 else (f(65504.0) if np.isinf(s) else s)
        elif kind == "content":
            s = torch.tensor(s).to(torch.bfloat16).float().numpy().astype(f)[()]
        clip = lambda v: np.fmin(np.fmax(v, f(0)), m)  # noqa: E731
        z = clip(np.rint(f(-lo / s)))
        return clip(np.rint((x / s).astype(f) + z)).astype(np.int64), s, z


@pytest.mark.parametrize("kind", [4, 2, "c4r4"])
def test_infinite_and_nan_values(kind):
    x = torch.randn(12, 9, 64, generator=torch.Generator().manual_seed(3))
    x[0, :, 5] = float("inf")
    x[1, :, 5] = -float("inf")
    x[2, :, 3], x[2, :, 9] = float("inf"), -float("inf")
    x[3, :, ::2] = float("nan")
    x[4] = float("nan")
    x[5] = float("inf")
    x[6, :, 7], x[6, :, 8] = 3e38, -3e38
    x[7] *= 1e-39
    x[8, :, 0], x[8, :, 1] = float("nan"), float("inf")
    x[9] = x[9] * 1e-4 + 1.0
    x[10, :, 63] = 2e38
    x = x.to(torch.bfloat16)
    lat, kpe = x[:, :8].reshape(12, 512).contiguous(), x[:, 8].contiguous()
    got, table = _append(kind, lat, kpe, 0)
    page = got[table[0][0]]
    for t in range(12):
        for g in range(9):
            bits = 4 if g == 8 or kind == "c4r4" else kind
            how = "own" if kind != "c4r4" else ("content" if g < 8 else "rope")
            q, s, z = _group(x[t, g].float().numpy(), bits, how)
            cb = 64 * (4 if kind == "c4r4" else kind) // 8
            off = g * 64 * cb + t * cb if g < 8 else 8 * 64 * cb + t * 32
            raw = page[off:off + 8 * bits].astype(np.int64)
            per = 8 // bits
            codes = np.stack([(raw >> (bits * i)) & (2 ** bits - 1) for i in range(per)], 1).reshape(-1)
            assert np.array_equal(codes, q), (t, g)
            if kind != "c4r4":
                at = 8 * 64 * cb + 2048 + (g * 64 + t) * 4
                sz = page[at:at + 4].view(np.float16).astype(np.float32)
                assert (sz[0], sz[1]) == (s, z), (t, g)
            else:
                assert page[19712 + g * 64 + t] == z, (t, g)
