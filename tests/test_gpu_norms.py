"""The value norms that ride in the tensor-core scoring passes: half of a sequence's rows in each
pass, cut into chunks of 4 KB per warp.  Lengths around the chunk, share and tile edges."""
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
@pytest.mark.parametrize("lens,heads", [((33, 64), (2, 1)), ((255, 257), (4, 4)), ((1023, 2049, 777), (8, 2)),
                                        ((8191,), (2, 2)), ((4097, 300), (16, 1))])
def test_norms_of_the_scoring_passes(d, lens, heads):
    hq, hkv = heads
    n, W = max(lens), 32
    g = torch.Generator(device="cuda").manual_seed(sum(lens) + d)
    K, V = (torch.randn((len(lens), hkv, n, d), generator=g, device="cuda").bfloat16() for _ in range(2))
    V *= torch.rand((len(lens), hkv, n, 1), generator=g, device="cuda").bfloat16() * 8
    Q = torch.randn((len(lens), hq, W, d), generator=g, device="cuda").bfloat16()
    shape = api.make_shape("bf16", len(lens), hq, hkv, d, W, n, api.capacity(n, 0.5))
    cache = api.compress(shape, lens, 0.5, K, V, Q, S.selkv_params.defaults(pool_kernel=1, recent=0), debug=True)
    torch.cuda.synchronize()
    for b, nb in enumerate(lens):
        # without pooling the score is a ||v||.  In fp32: a sum of d squares over 8 terms in a
        # lane and 4 butterfly levels, a root and two products: under 9 roundings of 2^-24
        want = cache.debug["attn"][b, :, :nb].double() * V[b, :, :nb].double().norm(dim=2)
        got = cache.debug["score"][b, :, :nb].double()
        np.testing.assert_allclose(got.cpu().numpy(), want.cpu().numpy(), rtol=9 * 2.0 ** -24, atol=0)
