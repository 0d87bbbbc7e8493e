"""The tensor-core scoring's shares of key tiles, against plain torch in 64 bits: every unit cut into
equal splits, shares that cross from one (sequence, KV head) to the next, several whole units in a
share, and each number of row halves.  Without pooling the score is a ||v||, so the value norms, which
follow the same shares, are checked too."""
import math

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
@pytest.mark.parametrize("lens,hq,hkv,W", [
    ((40,), 1, 1, 33),                       # one tile
    ((20000,), 16, 4, 64),                   # splits of one length
    ((9000, 257, 4100), 8, 4, 64),           # crossings, unequal lengths
    ((3001,) * 3, 32, 32, 32),               # units that do not divide the SMs
    ((129, 1, 256, 300) * 75, 2, 1, 1),      # more units than SMs, several in a share
    ((700, 5000) * 20, 16, 8, 40),           # 80 rows
    ((6000, 513), 12, 2, 64),                # 384 rows: three row parts of pass 1
    ((2500, 8000, 64), 16, 2, 64),           # 512 rows
])
def test_scores(d, lens, hq, hkv, W):
    B, n, G = len(lens), max(lens), hq // hkv
    g = torch.Generator(device="cuda").manual_seed(n + hq + d)
    K, V = (torch.randn((B, hkv, n, d), generator=g, device="cuda").bfloat16() for _ in range(2))
    Q = torch.randn((B, hq, W, d), generator=g, device="cuda").bfloat16()
    shape = api.make_shape("bf16", B, hq, hkv, d, W, n, api.capacity(n, 1.0))
    ws = api.Workspace(S.selkv_compress_workspace_size(shape))
    c = api.compress(shape, lens, 1.0, K, V, Q, S.selkv_params.defaults(recent=0, pool_kernel=1), debug=True, workspace=ws)
    torch.cuda.synchronize()
    assert ws.errors() == 0
    for b, nb in enumerate(lens):
        vis = torch.arange(nb, device="cuda")[None] <= (nb - W + torch.arange(W, device="cuda"))[:, None]
        s = torch.einsum("hwd,hnd->hwn", Q[b].double(), K[b, :, :nb].double().repeat_interleave(G, 0)) / math.sqrt(d)
        want = torch.softmax(s.masked_fill(~vis, -math.inf), 2).sum(1).view(hkv, G, nb).mean(1)
        # the tolerance of the parity tests for `a`: fp32 sums of exponentials of rounded logits
        torch.testing.assert_close(c.debug["attn"][b, :, :nb].double(), want, rtol=5e-5, atol=1e-12)
        want = c.debug["attn"][b, :, :nb].double() * V[b, :, :nb].double().norm(dim=2)
        torch.testing.assert_close(c.debug["score"][b, :, :nb].double(), want, rtol=9 * 2.0 ** -24, atol=0)


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("lens,hq,hkv,W", [((9000, 257, 4100), 8, 4, 64), ((700, 5000) * 20, 16, 8, 40), ((2500, 8000, 64), 16, 2, 64)])
def test_column_sums_alone_keep_the_lengths_of_the_row_statistics(lens, hq, hkv, W, dtype):
    """A call with the second pass alone works on the lengths of the call before, whatever valid
    lengths it is given itself."""
    B, n, d = len(lens), max(lens), 64
    g = torch.Generator(device="cuda").manual_seed(n)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    K = torch.randn((B, hkv, n, d), generator=g, device="cuda").to(dt)
    Q = torch.randn((B, hq, W, d), generator=g, device="cuda").to(dt)
    shape = api.make_shape(dtype, B, hq, hkv, d, W, n, 64)
    ws = api.Workspace(S.selkv_score_workspace_size(shape))
    want = torch.full((B, hkv, n), -1.0, device="cuda")
    S.check(S.selkv_score(shape, lens, K, Q, want, S.SELKV_SCORE_ALL, ws.buf, ws.nbytes), "all")
    for other in (lens, [W] * B, [n] * B, list(reversed(lens))):
        got = torch.full_like(want, -1.0)
        S.check(S.selkv_score(shape, lens, K, Q, None, S.SELKV_SCORE_ROWSTATS, ws.buf, ws.nbytes), "rowstats")
        S.check(S.selkv_score(shape, other, K, Q, got, S.SELKV_SCORE_COLSUMS, ws.buf, ws.nbytes), "colsums")
        assert torch.equal(got, want)
    assert ws.errors() == 0
