"""Calls on the default stream, where kernels are brought up before their predecessor has finished: several
compressions on one workspace, each followed at once by a decode of its cache, with nothing between
them that waits for the device.  They give, bit for bit, what the same calls give on a stream of
their own, where each kernel starts after the one before, with a wait after every call."""
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


# caches of 1500 rows and 160 units: the decode starts on whole tiles of them early
@pytest.mark.parametrize("dtype,B,n,opts", [
    ("bf16", 20, 5000, {}),
    ("bf16", 20, 5000, dict(select_mode=S.SELKV_SELECT_PER_HEAD)),
    ("bf16", 20, 5000, dict(rope=S.SELKV_ROPE_HALF)),
    ("bf16", 20, 5000, dict(bucket=16)),
    ("bf16", 2, 3000, dict(routing=S.SELKV_ROUTE_COSINE)),
    ("bf16", 1, 40000, {}),
    ("fp32", 2, 1500, {}),
    ("fp32", 2, 1500, dict(select_mode=S.SELKV_SELECT_PER_HEAD, rope=S.SELKV_ROPE_HALF)),
])
def test_early_starts_change_nothing(dtype, B, n, opts):
    hq, hkv, d, W, rho = 16, 8, 128, 32, 0.3
    g = torch.Generator(device="cuda").manual_seed(n)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    lens = [n - 7 * b for b in range(B)]
    shape = api.make_shape(dtype, B, hq, hkv, d, W, n, api.capacity(n, rho))
    params = S.selkv_params.defaults(**opts)
    layers = []
    for _ in range(3):
        K, V = (torch.randn((B, hkv, n, d), generator=g, device="cuda").to(dt) for _ in range(2))
        layers.append((K, V, torch.randn((B, hq, W, d), generator=g, device="cuda").to(dt)))
    q = torch.randn((B, hq, d), generator=g, device="cuda").to(dt)
    torch.cuda.synchronize()  # the inputs exist before another stream reads them

    def run(stream, wait):
        handle = stream.cuda_stream
        with torch.cuda.stream(stream):
            ws = api.Workspace(S.selkv_compress_workspace_size(shape), "cuda", handle)
            wd = api.Workspace(S.selkv_decode_workspace_size(shape), "cuda", handle)
            caches = [api.alloc_compressed(shape) for _ in layers]
            outs = [torch.empty_like(q) for _ in layers]
            torch.cuda.synchronize()
            for x, c, o in zip(layers, caches, outs):
                api.compress(shape, lens, rho, *x, params=params, out=c, workspace=ws, stream=handle)
                if wait:
                    torch.cuda.synchronize()
                api.decode(c, q, out=o, workspace=wd, stream=handle)
                if wait:
                    torch.cuda.synchronize()
            torch.cuda.synchronize()
            assert ws.errors(handle) == 0 and wd.errors(handle) == 0
        return [(c.K_c, c.V_c, c.bias, c.lengths, o) for c, o in zip(caches, outs)]

    early, plain = run(torch.cuda.default_stream(), False), run(torch.cuda.Stream(), True)
    assert torch.cuda.default_stream().cuda_stream == 0
    for a, b in zip(early, plain):
        for x, y in zip(a, b):
            assert torch.equal(x, y)
