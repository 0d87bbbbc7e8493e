"""Decode of many short caches, whose units the CTAs walk longest first: ragged and equal lengths, empty
and full caches, more sequences than one warp's lanes, several tokens in a row (the lengths advance
once per token), against plain torch in 64 bits."""
import math

import pytest
import torch

from paper_2607_16213_gb300 import api
import paper_2607_16213_gb300 as S

from parity import DEC_BF16_MAX, DEC_BF16_MEAN

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2607_16213_gb300 import build as b
    b.build()
    S.library()


@pytest.mark.parametrize("B,hq,hkv,d,cap,lens", [
    (64, 32, 8, 128, 896, "ragged"), (33, 16, 8, 64, 256, "ragged"), (160, 1, 1, 128, 192, "equal"),
    (300, 8, 2, 128, 128, "ragged"), (77, 32, 2, 64, 2112, "ragged"), (1000, 4, 1, 64, 64, "edges"),
    (40, 8, 4, 128, 320, "edges")])
def test_tokens(B, hq, hkv, d, cap, lens):
    g = torch.Generator(device="cuda").manual_seed(B + cap)
    if lens == "ragged":
        n = torch.randint(1, cap - 4, (B,), generator=g, device="cuda")
    elif lens == "equal":
        n = torch.full((B,), cap - 5, device="cuda")
    else:  # around the 64-row steps, empty, and full but for one row
        n = torch.tensor([0, 1, 63, 64, 65, cap - 4, cap - 1], device="cuda").clamp(max=cap - 1)[torch.arange(B, device="cuda") % 7]
    n = n.int()
    K, V = (torch.randn((B, hkv, cap, d), generator=g, device="cuda").bfloat16() for _ in range(2))
    bias = torch.rand((B, hkv, cap), generator=g, device="cuda")
    shape = api.make_shape("bf16", B, hq, hkv, d, 32, cap, cap)
    lengths = torch.zeros(((B + 3) // 4 * 4,), dtype=torch.int32, device="cuda")
    lengths[:B] = n
    cache = api.CompressedCache(shape, K, V, bias, lengths)
    ws = api.Workspace(S.selkv_decode_workspace_size(shape))
    col = torch.arange(cap, device="cuda")
    for token in range(3):
        q = torch.randn((B, hq, d), generator=g, device="cuda").bfloat16()
        kn, vn = (torch.randn((B, hkv, d), generator=g, device="cuda").bfloat16() for _ in range(2))
        app = n + 1 <= cap
        out = api.decode(cache, q, kn, vn, workspace=ws)
        torch.cuda.synchronize()
        # the row appended by this token is in the cache now, with bias 0
        rows = torch.where(app, n + 1, n)
        s = torch.einsum("bkgd,bknd->bkgn", q.view(B, hkv, hq // hkv, d).double(), K.double()) / math.sqrt(d)
        s = (s + bias.double()[:, :, None]).masked_fill((col[None] >= rows[:, None])[:, None, None], -math.inf)
        want = torch.einsum("bkgn,bknd->bkgd", torch.softmax(s, 3), V.double()).reshape(B, hq, d)
        err = (out.double() - want).abs()
        assert float(err.max()) <= DEC_BF16_MAX and float(err.mean()) <= DEC_BF16_MEAN
        at = n.long().clamp(max=cap - 1)
        b = torch.arange(B, device="cuda")
        assert torch.equal(K[b, :, at][app], kn[app]) and torch.equal(V[b, :, at][app], vn[app])
        n = rows.int()
        assert torch.equal(lengths[:B], n)
        assert ws.errors() == (0 if bool(app.all()) else S.SELKV_DEVERR_CAPACITY)


@pytest.mark.parametrize("hq,hkv,d", [(32, 8, 128), (128, 8, 128), (16, 8, 64)])
def test_the_output_does_not_depend_on_the_tile(hq, hkv, d):
    """Up to 304 units of more than 1024 rows are walked in 128-row tiles, more of them in 64-row
    tiles: the same sequences, once alone and once among copies of themselves, give the same bits."""
    B, cap = 20, 1088
    g = torch.Generator(device="cuda").manual_seed(hq + d)
    K, V = (torch.randn((B, hkv, cap, d), generator=g, device="cuda").bfloat16() for _ in range(2))
    bias = torch.rand((B, hkv, cap), generator=g, device="cuda")
    n = torch.randint(1, cap - 1, (B,), generator=g, device="cuda").int()
    n[:7] = torch.tensor([1, 16, 64, 65, 128, 129, cap - 1])
    q = torch.randn((B, hq, d), generator=g, device="cuda").bfloat16()
    kn, vn = (torch.randn((B, hkv, d), generator=g, device="cuda").bfloat16() for _ in range(2))
    outs = []
    for copies in (1, 2):
        both = [x.repeat(copies, *[1] * (x.dim() - 1)) for x in (K, V, bias, n, q, kn, vn)]
        shape = api.make_shape("bf16", B * copies, hq, hkv, d, 32, cap, cap)
        cache = api.CompressedCache(shape, *both[:4])
        outs.append(api.decode(cache, *both[4:]))
    assert torch.equal(outs[1][:B], outs[0]) and torch.equal(outs[1][B:], outs[0])


@pytest.mark.parametrize("B,hkv,full", [(1000, 1, 0), (1000, 1, 3), (90, 8, 40), (20, 8, 0)])
def test_many_empty_caches(B, hkv, full):
    """All but `full` caches are empty, several for each CTA: no consumer waits for a tile of theirs.
    Three tokens in a row, with nothing between them that waits for the device."""
    d, cap = 64, 192
    g = torch.Generator(device="cuda").manual_seed(B + full)
    K, V = (torch.randn((B, hkv, cap, d), generator=g, device="cuda").bfloat16() for _ in range(2))
    bias = torch.rand((B, hkv, cap), generator=g, device="cuda")
    lengths = torch.zeros(((B + 3) // 4 * 4,), dtype=torch.int32, device="cuda")
    lengths[:full] = cap - 3
    shape = api.make_shape("bf16", B, 2 * hkv, hkv, d, 32, cap, cap)
    cache = api.CompressedCache(shape, K, V, bias, lengths)
    ws = api.Workspace(S.selkv_decode_workspace_size(shape))
    q = torch.randn((3, B, 2 * hkv, d), generator=g, device="cuda").bfloat16()
    kn, vn = (torch.randn((3, B, hkv, d), generator=g, device="cuda").bfloat16() for _ in range(2))
    outs = [api.decode(cache, q[t], kn[t], vn[t], workspace=ws) for t in range(3)]
    assert ws.errors() == 0
    assert torch.equal(lengths[:B], (torch.arange(B, device="cuda") < full).int() * (cap - 3) + 3)
    assert torch.equal(K[full:, :, :3], kn[:, full:].permute(1, 2, 0, 3)) and torch.equal(V[full:, :, :3], vn[:, full:].permute(1, 2, 0, 3))
    # one row: its value; then a softmax over the rows so far, all with bias 0
    assert torch.equal(outs[0][full:], vn[0, full:].repeat_interleave(2, 1))
    for t in range(1, 3):
        s = torch.einsum("bkgd,tbkd->bkgt", q[t, full:].view(-1, hkv, 2, d).double(), kn[:t + 1, full:].double()) / math.sqrt(d)
        want = torch.einsum("bkgt,tbkd->bkgd", torch.softmax(s, 3), vn[:t + 1, full:].double()).reshape(-1, 2 * hkv, d)
        assert float((outs[t][full:].double() - want).abs().max()) <= DEC_BF16_MAX
