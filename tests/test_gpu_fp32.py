"""fp32 caches on the CUDA cores, against plain torch in 64 bits: scoring over every width of its
column chunks (64 to 512), and decode around the edges of a warp's step and of a split."""
import math

import numpy as np
import pytest
import torch

from paper_2607_16213_gb300 import api
import paper_2607_16213_gb300 as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2607_16213_gb300 import build as b
    b.build()
    S.library()


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("lens,hq,hkv,W", [((33,), 2, 2, 32), ((65, 64), 4, 2, 32), ((1500,), 4, 2, 32), ((2049, 300), 16, 8, 32),
                                           ((700,) * 12, 8, 8, 16), ((1100,) * 40, 4, 4, 16), ((3000,), 20, 2, 20)])
def test_scoring(d, lens, hq, hkv, W):
    B, n, G = len(lens), max(lens), hq // hkv
    g = torch.Generator(device="cuda").manual_seed(n + hq + d)
    K, V = (torch.randn((B, hkv, n, d), generator=g, device="cuda") for _ in range(2))
    Q = torch.randn((B, hq, W, d), generator=g, device="cuda")
    shape = api.make_shape("fp32", B, hq, hkv, d, W, n, api.capacity(n, 0.5))
    c = api.compress(shape, lens, 0.5, K, V, Q, S.selkv_params.defaults(recent=0), debug=True)
    for b, nb in enumerate(lens):
        vis = torch.arange(nb, device="cuda")[None] <= (nb - W + torch.arange(W, device="cuda"))[:, None]
        s = torch.einsum("hwd,hnd->hwn", Q[b].double(), K[b, :, :nb].double().repeat_interleave(G, 0)) / math.sqrt(d)
        want = torch.softmax(s.masked_fill(~vis, -math.inf), 2).sum(1).view(hkv, G, nb).mean(1)
        # logits of d products of up to ~4 sqrt(d): their rounding (2^-24 sqrt(d) of it) goes into the exponent
        torch.testing.assert_close(c.debug["attn"][b, :, :nb].double(), want, rtol=2e-5, atol=1e-9)


@pytest.mark.parametrize("append", [False, True])
@pytest.mark.parametrize("d,hq,hkv", [(64, 4, 2), (128, 3, 1), (64, 8, 8), (128, 16, 2), (64, 16, 1)])
@pytest.mark.parametrize("lens", [(1,), (7, 8, 9), (63, 64, 65), (127, 129), (320,), (2000, 1)])
def test_decode(lens, d, hq, hkv, append):
    B, cap, G = len(lens), (max(lens) + 64) // 64 * 64, hq // hkv
    g = torch.Generator(device="cuda").manual_seed(sum(lens) + d + hq)
    K, V = (torch.randn((B, hkv, cap, d), generator=g, device="cuda") for _ in range(2))
    bias = torch.rand((B, hkv, cap), generator=g, device="cuda")
    q = torch.randn((B, hq, d), generator=g, device="cuda")
    kn, vn = (torch.randn((B, hkv, d), generator=g, device="cuda") for _ in range(2))
    lengths = torch.zeros(((B + 3) // 4 * 4,), dtype=torch.int32, device="cuda")
    lengths[:B] = torch.tensor(lens, dtype=torch.int32)
    for b, nb in enumerate(lens):  # rows past the length are never used
        K[b, :, nb:], V[b, :, nb:], bias[b, :, nb:] = math.nan, math.nan, math.nan
    shape = api.make_shape("fp32", B, hq, hkv, d, 32, cap, cap)
    cache = api.CompressedCache(shape, K, V, bias, lengths)
    out = api.decode(cache, q, kn if append else None, vn if append else None)
    for b, nb in enumerate(lens):
        Kb, Vb, bb = K[b, :, :nb].double(), V[b, :, :nb].double(), bias[b, :, :nb].double()
        if append:
            Kb, Vb = torch.cat([Kb, kn[b, :, None].double()], 1), torch.cat([Vb, vn[b, :, None].double()], 1)
            bb = torch.cat([bb, torch.zeros_like(bb[:, :1])], 1)
            torch.testing.assert_close(K[b, :, nb], kn[b], rtol=0, atol=0)
        s = torch.einsum("kgd,knd->kgn", q[b].view(hkv, G, d).double(), Kb) / math.sqrt(d) + bb[:, None]
        want = torch.einsum("kgn,knd->kgd", torch.softmax(s, 2), Vb).reshape(hq, d)
        # fp32 sums of at most 2000 terms of order 1 in a tree over warps: well under 1e-5 of the largest
        assert float((out[b].double() - want).abs().max()) <= 1e-5 * max(1.0, float(want.abs().max()))
        assert int(lengths[b]) == nb + append
    np.testing.assert_equal(lengths[B:].cpu().numpy(), 0)


@pytest.mark.parametrize("append", [False, True])
@pytest.mark.parametrize("d,hq,hkv", [(64, 4, 2), (128, 4, 2), (128, 16, 1)])
@pytest.mark.parametrize("masked", [(0, 1), (0, 8), (0, 16), (0, 32), (0, 64), (0, 255), (64, 128), (3, 300)])
def test_decode_of_rows_masked_by_the_bias(masked, d, hq, hkv, append):
    """A bias of -inf takes a row out, also where it does so for all rows of a warp's step (8 at d 128, 16
    at d 64), of a warp or of a split."""
    cap, n, G = 384, 320, hq // hkv
    g = torch.Generator(device="cuda").manual_seed(sum(masked) + d)
    K, V = (torch.randn((1, hkv, cap, d), generator=g, device="cuda") for _ in range(2))
    bias = torch.rand((1, hkv, cap), generator=g, device="cuda")
    bias[:, :, masked[0]:masked[1]] = -math.inf
    q = torch.randn((1, hq, d), generator=g, device="cuda")
    kn, vn = (torch.randn((1, hkv, d), generator=g, device="cuda") for _ in range(2))
    lengths = torch.tensor([n, 0, 0, 0], dtype=torch.int32, device="cuda")
    cache = api.CompressedCache(api.make_shape("fp32", 1, hq, hkv, d, 32, cap, cap), K, V, bias, lengths)
    out = api.decode(cache, q, kn if append else None, vn if append else None)
    rows = n + append  # (an appended row is in the cache now, with bias 0)
    s = torch.einsum("kgd,knd->kgn", q[0].view(hkv, G, d).double(), K[0, :, :rows].double()) / math.sqrt(d)
    s = s + bias[0, :, None, :rows].double()
    want = torch.einsum("kgn,knd->kgd", torch.softmax(s, 2), V[0, :, :rows].double()).reshape(hq, d)
    # fp32 sums of a few hundred terms of order 1, as above
    assert float((out[0].double() - want).abs().max()) <= 1e-5 * max(1.0, float(want.abs().max()))
