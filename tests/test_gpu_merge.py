"""The one-kernel merge of bf16 caches with 32-token buckets, against the oracle: lengths around the
edges of a bucket and of a warp's walk, buckets without a kept token (tight budgets), both head
sizes, and rows that are not finite."""
import functools

import numpy as np
import pytest
import torch

import synth
from oracle import selkv_oracle as O
from paper_2607_16213_gb300 import api
import paper_2607_16213_gb300 as S

from parity import check_sequence, params_of, run_compress, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2607_16213_gb300 import build as b
    b.build()
    S.library()


def workload(n, d=128, heads=(8, 2), batch=2, rho=0.25):
    return synth.WORKLOADS["llama_layer"].with_(name="merge_%d" % n, batch=batch, n=n, head_dim=d, num_q_heads=heads[0],
                                                num_kv_heads=heads[1], obs_window=24, rho=rho, ragged=(0.6, 1.0), seed=n)


@pytest.mark.parametrize("mode", ["shared", "per_head", "rope", "rope_pairs", "drop"])
@pytest.mark.parametrize("n,d,rho", [(64, 128, 0.5), (65, 64, 0.3), (95, 128, 0.3), (257, 64, 0.1), (2049, 128, 0.02),
                                     (4000, 128, 0.008), (4000, 64, 0.6)])
def test_merge_matches_the_oracle(n, d, rho, mode):
    wl = workload(n, d, rho=rho, batch=1 if n >= 4000 else 2)
    p = O.Params(recent=min(16, int(0.5 * rho * wl.n * 0.6)),
                 select_mode=O.SELECT_PER_HEAD if mode == "per_head" else O.SELECT_SHARED,
                 rope={"rope": O.ROPE_HALF, "rope_pairs": O.ROPE_INTERLEAVED}.get(mode, O.ROPE_OFF),
                 empty_bucket=O.EMPTY_DROP if mode == "drop" else O.EMPTY_EXPAND)
    x = synth.gen_layer(wl, 0)
    _, host, _ = run_compress(wl, x, p)
    for b in range(wl.batch):
        check_sequence(wl, x, host, b, p)


def test_long_walks_match_the_oracle():
    """Enough buckets that a warp walks its longest range."""
    wl = workload(26000, 64, heads=(16, 16), batch=1, rho=0.05).with_(ragged=None)
    p = O.Params()
    x = synth.gen_layer(wl, 0)
    _, host, _ = run_compress(wl, x, p)
    check_sequence(wl, x, host, 0, p)


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_a_kept_row_that_is_not_finite_stays_where_it_is(bad):
    """Such a row is copied; the rows merged in its bucket are as without it."""
    wl = workload(1000, batch=1).with_(ragged=None)
    p = O.Params()
    x = synth.gen_layer(wl, 0)
    _, host, (K, V, Q) = run_compress(wl, x, p)
    targets = set(host["target"][0].ravel().tolist())
    pos = next(j for j in range(wl.n - 1, wl.n - p.recent - 1, -1) if j not in targets)
    m = int(host["lengths"][0])
    slot = int(np.flatnonzero(host["kept_idx"][0, :m] == pos)[0])
    V2 = V.clone()
    V2[0, :, pos, 3] = bad
    shape = api.make_shape("bf16", 1, wl.num_q_heads, wl.num_kv_heads, wl.head_dim, wl.obs_window, wl.n,
                           host["V_c"].shape[2])
    c = api.compress(shape, [wl.n], wl.rho, K, V2, Q, params=params_of(p))
    torch.cuda.synchronize()
    got = c.V_c[0, :, :m].float().cpu().numpy()
    others = np.arange(m) != slot
    np.testing.assert_array_equal(got[:, others], host["V_c"][0, :, :m][:, others])
    np.testing.assert_array_equal(got[:, slot], V2[0, :, pos].float().cpu().numpy())


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_the_same_with_the_gate_open(bad, monkeypatch):
    """Without the cosines nothing comes between the copy of the row and its clearing in the tile."""
    monkeypatch.setattr(O, "Params", functools.partial(O.Params, gate_mode=O.GATE_OPEN))
    test_a_kept_row_that_is_not_finite_stays_where_it_is(bad)


@pytest.mark.parametrize("d", [64, 128])
def test_the_smallest_weights_keep_their_bits(d):
    """All tokens but one have an attention of 2^-120 to 2^-125, close to the smallest normal number: the
    merged values are still the exact ones rounded to bf16."""
    n, W, m_r = 2000, 1, 16
    g = torch.Generator(device="cuda").manual_seed(d)
    V = torch.randn((1, 1, n, d), generator=g, device="cuda").bfloat16()
    V[..., 0] = 4.0  # cosines well above 0
    K = torch.zeros((1, 1, n, d), device="cuda")
    Q = torch.zeros((1, 1, W, d), device="cuda")
    Q[..., 0] = 8.0
    # one key takes all of the attention
    K[..., 0] = -(120.0 + 4.5 * torch.rand((1, 1, n), generator=g, device="cuda")) * float(np.log(2.0)) * d ** 0.5 / 8.0
    K[0, 0, n // 2, 0] = 0.0
    K, Q = K.bfloat16(), Q.bfloat16()
    shape = api.make_shape("bf16", 1, 1, 1, d, W, n, 576)
    c = api.compress(shape, [n], 0.25, K, V, Q, S.selkv_params.defaults(recent=m_r), debug=True)
    m = int(c.lengths[0])
    a = c.debug["attn"][0, 0, :n].double().cpu().numpy()
    small = a[:n - W]
    assert np.median(small) < 2.0 ** -121 and (small > 0).mean() > 0.9
    kept, target = (c.debug[k][0, 0].cpu().numpy() if c.debug[k].dim() == 3 else c.debug[k][0].cpu().numpy()
                    for k in ("kept_idx", "target"))
    kept, gate = kept[:m], c.debug["gate"][0, 0].double().cpu().numpy()
    v = V[0, 0].double().cpu().numpy()
    num, den = a[kept, None] * v[kept], a[kept].copy()
    slot = {int(p): i for i, p in enumerate(kept)}
    for j in range(n):
        if target[j] >= 0:
            num[slot[target[j]]] += gate[j] * a[j] * v[j]
            den[slot[target[j]]] += gate[j] * a[j]
    ok = den > 0
    want = num[ok] / den[ok, None]
    got = c.V_c[0, 0, :m].double().cpu().numpy()[ok]
    # half a unit in the last place of bf16, and fp32 sums of tens of terms up to 4 (g a below 2^-126
    # loses up to 2^-23 of itself as a subnormal number)
    half_ulp = 2.0 ** (np.floor(np.log2(np.maximum(np.abs(want), 2.0 ** -100))) - 8)
    assert (np.abs(got - want) - half_ulp).max() <= 1e-5
