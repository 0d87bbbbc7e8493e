"""Cosine routing's argmax around the edges of its tiles (256 evicted rows in two halves of 128, 256 kept
slots), against plain torch in 64 bits: every target is within rounding of the best cosine."""
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
@pytest.mark.parametrize("n,m", [(40, 32), (256, 127), (257, 128), (385, 129), (512, 256), (513, 256), (900, 257),
                                 (3000, 1100), (2600, 2343)])
def test_targets(n, m, d):
    hkv, W = 2, 32
    g = torch.Generator(device="cuda").manual_seed(n + m + d)
    K, V = (torch.randn((1, hkv, n, d), generator=g, device="cuda").bfloat16() for _ in range(2))
    Q = torch.randn((1, 2 * hkv, W, d), generator=g, device="cuda").bfloat16()
    rho = (m + 0.5) / n
    shape = api.make_shape("bf16", 1, 2 * hkv, hkv, d, W, n, api.capacity(n, rho))
    ws = api.Workspace(S.selkv_compress_workspace_size(shape))
    c = api.compress(shape, [n], rho, K, V, Q, S.selkv_params.defaults(recent=8, routing=S.SELKV_ROUTE_COSINE), debug=True,
                     workspace=ws)
    torch.cuda.synchronize()
    assert ws.errors() == 0 and int(c.lengths[0]) == m
    kept = c.debug["kept_idx"][0, :m].long()
    mask = torch.zeros(n, dtype=torch.bool, device="cuda")
    mask[kept] = True
    for h in range(hkv):
        v = V[0, h].double()
        v = v / v.norm(dim=1, keepdim=True)
        cos = v[~mask] @ v[kept].T
        target = c.debug["target"][0, h][~mask].long()
        assert bool(mask[target].all())
        got = (v[~mask] * v[target]).sum(1)
        # fp32 sums of d exact products and one scaling: a few 2^-24 sqrt(d)
        assert float((cos.max(1).values - got).max()) <= 2e-6
        gate = c.debug["gate"][0, h][~mask].double()
        assert float((gate - got.clamp(0, 1)).abs().max()) <= 2e-6
