"""The clustered selection against a plain top-k of its own scores: the decisions depend on the
scores' bits alone, so every set must agree exactly.  Sizes around the spans of a cluster's CTAs,
keys held in shared memory and (a very long sequence) in global memory, and scores with long runs of
ties, which the position decides."""
import numpy as np
import pytest
import torch

from paper_2607_16213_gb300 import api
import paper_2607_16213_gb300 as S

pytestmark = pytest.mark.gpu

RECENT, RHO = 16, 0.3


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2607_16213_gb300 import build as b
    b.build()
    S.library()


def top(key, member, k):
    """The k largest of key among the members, ties to the lower position."""
    cand = np.flatnonzero(member)
    order = cand[np.argsort(-key[cand].astype(np.float64), kind="stable")]
    out = np.zeros(key.shape[0], dtype=bool)
    out[order[:max(0, k)]] = True
    return out


@pytest.mark.parametrize("tied", [False, True])
@pytest.mark.parametrize("per_head", [False, True])
@pytest.mark.parametrize("hkv,lens,pool", [(2, (97,), 5), (8, (1023,), 5), (8, (8193,), 5), (9, (16385, 12000), 3),
                                           (3, (4097, 2048, 5000), 1), (2, (700,) * 40, 5), (1, (400001,), 5),
                                           (8, (54,), 5)])
def test_selection_matches_a_plain_top_k(hkv, lens, pool, per_head, tied):
    B, n, d, W = len(lens), max(lens), 64, 32
    g = torch.Generator(device="cuda").manual_seed(n + hkv)
    V = torch.randn((B, hkv, n, d), generator=g, device="cuda")
    if tied:  # equal keys: equal attention; the values take four norms, in runs
        K = torch.ones((B, hkv, n, d), device="cuda")
        level = torch.randint(1, 5, (B, hkv, (n + 63) // 64), generator=g, device="cuda").repeat_interleave(64, 2)
        V = torch.zeros_like(V)
        V[..., 0] = level[..., :n].float()
    else:
        K = torch.randn((B, hkv, n, d), generator=g, device="cuda")
    Q = torch.randn((B, hkv, W, d), generator=g, device="cuda")
    shape = api.make_shape("bf16", B, hkv, hkv, d, W, n, api.capacity(n, RHO))
    params = S.selkv_params.defaults(pool_kernel=pool, recent=RECENT,
                                     select_mode=S.SELKV_SELECT_PER_HEAD if per_head else S.SELKV_SELECT_SHARED)
    ws = api.Workspace(S.selkv_compress_workspace_size(shape))
    c = api.compress(shape, lens, RHO, K.bfloat16(), V.bfloat16(), Q.bfloat16(), params, debug=True, workspace=ws)
    torch.cuda.synchronize()
    assert ws.errors() == 0
    score, topk, kept_idx = (c.debug[k].cpu().numpy() for k in ("score", "topk", "kept_idx"))
    for b, nb in enumerate(lens):
        m, ncand = int(RHO * nb), nb - RECENT
        ms = m - RECENT
        key = score[b, :, :ncand]
        every = np.ones(ncand, dtype=bool)
        heads = np.stack([top(key[h], every, ms) for h in range(hkv)])
        np.testing.assert_array_equal(topk[b, :, :ncand].astype(bool), heads)
        assert not topk[b, :, ncand:nb].any()
        if per_head:
            want = [np.append(np.flatnonzero(heads[h]), np.arange(ncand, nb)) for h in range(hkv)]
            np.testing.assert_array_equal(kept_idx[b, :, :m], np.stack(want))
            continue
        total = np.zeros(ncand, dtype=np.float32)
        for h in range(hkv):
            total += key[h]
        union = heads.any(axis=0)
        chosen = top(total, union, ms) if union.sum() > ms else union
        np.testing.assert_array_equal(kept_idx[b, :m], np.append(np.flatnonzero(chosen), np.arange(ncand, nb)))


@pytest.mark.parametrize("per_head", [False, True])
@pytest.mark.parametrize("rho,recent", [(1.0, 16), (1.0, 0), (0.25, 1025)])
@pytest.mark.parametrize("hkv,n", [(8, 4101), (1, 4101)])
def test_every_candidate_or_none(hkv, n, rho, recent, per_head):
    """No threshold is searched for, so the compaction's counts are the first that the CTAs of a
    cluster tell each other (rho 1: all kept; m = recent: the recent window alone)."""
    d, W = 64, 32
    g = torch.Generator(device="cuda").manual_seed(n + hkv)
    K, V = (torch.randn((2, hkv, n, d), generator=g, device="cuda").bfloat16() for _ in range(2))
    Q = torch.randn((2, hkv, W, d), generator=g, device="cuda").bfloat16()
    shape = api.make_shape("bf16", 2, hkv, hkv, d, W, n, api.capacity(n, rho))
    params = S.selkv_params.defaults(recent=recent,
                                     select_mode=S.SELKV_SELECT_PER_HEAD if per_head else S.SELKV_SELECT_SHARED)
    ws = api.Workspace(S.selkv_compress_workspace_size(shape))
    c = api.compress(shape, [n, n], rho, K, V, Q, params, debug=True, workspace=ws)
    torch.cuda.synchronize()
    assert ws.errors() == 0
    m = int(rho * n)
    kept = c.debug["kept_idx"].cpu().numpy()[..., :m].reshape(-1, m)
    np.testing.assert_array_equal(kept, np.broadcast_to(np.arange(n - m, n), kept.shape))
    assert bool(c.debug["topk"][:, :, :n - recent].all()) == (rho == 1.0)
