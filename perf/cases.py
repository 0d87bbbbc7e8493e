"""The work a user of the SelKV library has it do, as measurable cases.

Two calls carry the library: `compress` once after a prefill, per layer, and `decode` once per
layer and generated token.  The cases run them through `paper_2607_16213_gb300.api` on device
tensors, with the output cache and the workspace kept across calls as a serving program keeps
them.  Decode over many layers is recorded once as a CUDA graph, as a token loop is in practice;
single small calls are made eagerly.

Inputs follow the segmented-centroid recipe of the repository's workloads (segments of 4-64
tokens around a random centroid, noise 0.1-0.8 per segment, 1% of the positions with keys x4,
ragged lengths of 50-100% in a batch), drawn on the device from the seed.
"""
import math

import torch

import paper_2607_16213_gb300 as S
from paper_2607_16213_gb300 import api

_LLAMA = dict(dtype="bf16", hq=32, hkv=8, d=128, w=64)
_OPTS = dict(per_head=False, cosine=False, rope=False)
_ALPHA, _POOL, _BUCKET, _RECENT, _THETA = 0.5, 5, 32, 16, 10000.0


def listed():
    def comp(name, batch, n, rho, shape=_LLAMA, ragged=False, **opts):
        return dict(name=name, kind="compress", batch=batch, n=n, rho=rho, ragged=ragged, **{**shape, **_OPTS, **opts})

    def dec(name, batch, m, spare, layers, steps, graph, shape=_LLAMA, ragged=False, bias=True):
        return dict(name=name, kind="decode", batch=batch, m=m, spare=spare, layers=layers, steps=steps, graph=graph,
                    ragged=ragged, bias=bias, **shape)

    tiny = dict(dtype="fp32", hq=4, hkv=2, d=64, w=32)
    return [
        # a short fp32 prompt of a small model: latency and launches are everything
        comp("compress_fp32_1k", 1, 1024, 0.25, tiny),
        # one layer of an 8B model after a 16k prompt, the ordinary single-user call
        comp("compress_16k", 1, 16384, 0.25),
        # the long-context setting, one layer at 100k tokens
        comp("compress_100k", 1, 100000, 0.25),
        # a serving batch of eight long prompts of unequal length
        comp("compress_b8_32k", 8, 32768, 0.25, ragged=True),
        # a serving batch of many short prompts, tight budget
        comp("compress_b64_8k", 64, 8192, 0.10, ragged=True),
        # a multi-head-attention model (32 KV heads), each head keeping its own tokens
        comp("compress_per_head_31k", 1, 31500, 0.25, dict(_LLAMA, hkv=32, w=32), per_head=True),
        # a 70B model's wide query group, kept keys turned to their new positions
        comp("compress_g8_rope_16k", 1, 16383, 0.25, dict(_LLAMA, hq=64), rope=True),
        # the exhaustive routing option, one layer at 16k
        comp("compress_cosine_16k", 1, 16384, 0.25, cosine=True),
        # sixteen tokens of a small fp32 model, call by call
        dec("decode_fp32_256", 1, 256, 64, 1, 16, False, tiny),
        # a token of the long-context setting, eight of its layers (a 100k prompt at 25%)
        dec("decode_25k", 1, 25000, 256, 8, 1, True),
        # a token of a large ragged batch over short caches, four layers
        dec("decode_b64_819", 64, 819, 64, 4, 1, True, ragged=True),
        # a token of eight ragged long caches at a loose budget, two layers
        dec("decode_b8_16k", 8, 16384, 64, 2, 1, True, ragged=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: batches up to 64, contexts up to 131072 (at most 480k tokens
    of an 8-KV-head layer in all for a compression), budgets of 10-50%, both types, every option at its usual rate."""
    kind = rng.choice(("compress", "compress", "decode"))
    fp32 = rng.random() < 0.15
    hq, hkv = rng.choice(((32, 8), (32, 8), (32, 8), (64, 8), (32, 32), (32, 4)))
    batch = rng.choice((1, 1, 2, 5, 8, 16, 33, 64))
    ragged = batch > 1
    if kind == "compress":
        rho = round(rng.uniform(0.1, 0.5), 3)
        if fp32:
            return dict(kind=kind, batch=rng.choice((1, 2, 3)), n=_log_int(rng, 300, 4000), rho=rho, ragged=False,
                        dtype="fp32", hq=4, hkv=2, d=rng.choice((64, 128)), w=32, **_OPTS)
        cosine = rng.random() < 0.1
        most = 20000 if cosine else 131072
        total = int((20000 if cosine else 480000) / max(hq / 32, hkv / 8))
        n = _log_int(rng, 700, max(701, min(most, total // batch)))
        batch = max(1, min(batch, total // n))
        opts = dict(per_head=hkv == 32 or rng.random() < 0.1, cosine=cosine, rope=rng.random() < 0.2)
        return dict(kind=kind, batch=batch, n=n, rho=rho, ragged=batch > 1, dtype="bf16", hq=hq, hkv=hkv,
                    d=rng.choice((128, 128, 128, 64)), w=rng.choice((32, 64)) if hq // hkv <= 8 else 32, **opts)
    if fp32:
        return dict(kind=kind, batch=rng.choice((1, 2, 3)), m=_log_int(rng, 64, 4000), spare=64, layers=1,
                    steps=rng.choice((1, 4, 16)), graph=False, ragged=False, bias=True, dtype="fp32", hq=4, hkv=2,
                    d=rng.choice((64, 128)), w=32)
    m = _log_int(rng, 100, min(100000, max(200, 1200000 // (batch * hkv))))
    return dict(kind=kind, batch=batch, m=m, spare=64, layers=rng.choice((1, 2, 4)), steps=rng.choice((1, 2)),
                graph=rng.random() < 0.7, ragged=ragged, bias=rng.random() < 0.85, dtype="bf16", hq=hq, hkv=hkv,
                d=rng.choice((128, 128, 128, 64)), w=64)


# ---- inputs ----------------------------------------------------------------------------------
def _dtype(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _segmented(g, units, n, d, dtype, scale=None, tensors=1):
    """`tensors` arrays [units][n][d] over one segmentation; the first one's rows times `scale`
    [units][n]."""
    outs = [torch.empty((units, n, d), dtype=dtype, device="cuda") for _ in range(tensors)]
    step = max(1, (1 << 26) // max(1, n * d))
    for u0 in range(0, units, step):
        u = min(step, units - u0)
        lens = torch.randint(4, 65, (u, n // 4 + 1), generator=g, device="cuda")
        ends = lens.cumsum(1)
        seg = torch.searchsorted(ends, torch.arange(n, device="cuda").expand(u, n).contiguous(), right=True)
        nseg = int(seg.max()) + 1
        sigma = 0.1 + 0.7 * torch.rand((u, nseg), generator=g, device="cuda")
        sig = sigma.gather(1, seg)
        for i, out in enumerate(outs):
            cent = torch.randn((u, nseg, d), generator=g, device="cuda")
            x = torch.randn((u, n, d), generator=g, device="cuda")
            x.mul_(sig[:, :, None]).add_(torch.gather(cent, 1, seg[:, :, None].expand(u, n, d)))
            if scale is not None and i == 0:
                x.mul_(scale[u0:u0 + u, :, None])
            out[u0:u0 + u] = x.to(dtype)
    return outs


def _lengths(case, seed, n):
    """Rows of each sequence: all n, or ragged in [n/2, n]; of the case's sizes alone (the same
    work for every seed)."""
    b = case["batch"]
    if not case["ragged"] or b == 1:
        return [n] * b
    lo = max(n // 2, min(n, 128))
    return [lo + ((i * 2654435761 + 12345) % 1000003) * (n - lo + 1) // 1000003 for i in range(b)]


def _compress_inputs(case, seed):
    B, Hq, Hkv, d, W, n = (case[k] for k in ("batch", "hq", "hkv", "d", "w", "n"))
    g = _generator(seed)
    lens = _lengths(case, seed, n)
    heavy = torch.rand((B, n), generator=g, device="cuda") < 0.01
    scale = 1.0 + 3.0 * heavy.float()
    K, V = _segmented(g, B * Hkv, n, d, _dtype(case), scale.repeat_interleave(Hkv, 0), 2)
    (Q,) = _segmented(g, B * Hq, W, d, _dtype(case))
    K, V, Q = K.view(B, Hkv, n, d), V.view(B, Hkv, n, d), Q.view(B, Hq, W, d)
    for b, nb in enumerate(lens):
        K[b, :, nb:] = 0
        V[b, :, nb:] = 0
    return K, V, Q, lens


def _decode_inputs(case, seed):
    """A cache as a compression leaves it: segmented rows, and a bias alpha ln R >= 0 that is the
    same for every KV head, positive on the slots that took merged tokens (about one in eight)."""
    B, Hq, Hkv, d, L, T = (case[k] for k in ("batch", "hq", "hkv", "d", "layers", "steps"))
    g = _generator(seed)
    cap = api.capacity(case["m"], 1.0, extra=case["spare"])
    K, V = _segmented(g, L * B * Hkv, cap, d, _dtype(case), None, 2)
    K, V = K.view(L, B, Hkv, cap, d), V.view(L, B, Hkv, cap, d)
    merged = torch.rand((L, B, 1, cap), generator=g, device="cuda") < 0.125
    ratio = 1.0 + torch.empty((L, B, 1, cap), device="cuda").exponential_(0.25, generator=g) * merged
    bias = (_ALPHA * torch.log(ratio)).expand(L, B, Hkv, cap).contiguous()
    base = torch.zeros((L, (B + 3) // 4 * 4), dtype=torch.int32, device="cuda")
    base[:, :B] = torch.tensor(_lengths(case, seed, case["m"]), dtype=torch.int32, device="cuda")
    q = torch.randn((T, L, B, Hq, d), generator=g, device="cuda").to(_dtype(case))
    kn = torch.randn((T, L, B, Hkv, d), generator=g, device="cuda").to(_dtype(case))
    vn = torch.randn((T, L, B, Hkv, d), generator=g, device="cuda").to(_dtype(case))
    return K, V, bias, base, q, kn, vn, cap


def _params(case):
    return S.selkv_params.defaults(
        alpha=_ALPHA, pool_kernel=_POOL, bucket=_BUCKET, recent=_RECENT, rope_theta=_THETA,
        select_mode=S.SELKV_SELECT_PER_HEAD if case["per_head"] else S.SELKV_SELECT_SHARED,
        routing=S.SELKV_ROUTE_COSINE if case["cosine"] else S.SELKV_ROUTE_BUCKET,
        rope=S.SELKV_ROPE_HALF if case["rope"] else S.SELKV_ROPE_OFF)


# ---- one pass --------------------------------------------------------------------------------
class _Compress:
    def __init__(self, case, seed):
        self.K, self.V, self.Q, self.lens = _compress_inputs(case, seed)
        self.rho, self.params = case["rho"], _params(case)
        m_cap = api.capacity(case["n"], case["rho"])
        self.shape = api.make_shape(case["dtype"], case["batch"], case["hq"], case["hkv"], case["d"], case["w"],
                                    case["n"], m_cap)
        self.out = api.alloc_compressed(self.shape)
        self.ws = api.Workspace(S.selkv_compress_workspace_size(self.shape))

    def run(self):
        c = api.compress(self.shape, self.lens, self.rho, self.K, self.V, self.Q, params=self.params, out=self.out,
                         workspace=self.ws)
        return dict(K_c=c.K_c, V_c=c.V_c, bias=c.bias, lengths=c.lengths)


class _Decode:
    """A token loop over the layers' caches: `steps` tokens, each appending its row in every
    layer.  The lengths go back to the prompt's first, as for another continuation of it."""

    def __init__(self, case, seed):
        self.K, self.V, self.bias, self.base, self.q, self.kn, self.vn, cap = _decode_inputs(case, seed)
        self.lengths = self.base.clone()
        B = case["batch"]
        self.use_bias = case["bias"]
        self.shape = api.make_shape(case["dtype"], B, case["hq"], case["hkv"], case["d"], case["w"], cap, cap)
        self.caches = [api.CompressedCache(self.shape, self.K[i], self.V[i], self.bias[i], self.lengths[i])
                       for i in range(case["layers"])]
        self.ws = api.Workspace(S.selkv_decode_workspace_size(self.shape))
        self.out = torch.empty_like(self.q)
        # views of each call's tensors, laid out once
        self.calls = [(c, self.q[t, i], self.kn[t, i], self.vn[t, i], self.out[t, i])
                      for t in range(case["steps"]) for i, c in enumerate(self.caches)]
        self.graph = None
        if case["graph"]:
            self.loop()
            torch.cuda.synchronize()
            self.graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(self.graph):
                self.loop()

    def loop(self):
        self.lengths.copy_(self.base)
        for cache, q, kn, vn, out in self.calls:
            api.decode(cache, q, kn, vn, use_bias=self.use_bias, out=out, workspace=self.ws)

    def run(self):
        if self.graph is not None:
            self.graph.replay()
        else:
            self.loop()
        return dict(out=self.out, lengths=self.lengths, K=self.K, V=self.V, bias=self.bias)


def prepare(case, seed):
    return (_Compress if case["kind"] == "compress" else _Decode)(case, seed)


def run(state):
    return state.run()


def work(case):
    e = 2 if case["dtype"] == "bf16" else 4
    B, Hq, Hkv, d = case["batch"], case["hq"], case["hkv"], case["d"]
    if case["kind"] == "compress":
        lens = _lengths(case, 0, case["n"])
        rows = sum(lens)
        kept = sum(int(case["rho"] * n) for n in lens)
        # K, V and Q_obs in; K_c, V_c and the bias out.  One product of the window with the keys
        # (the values' cosines are d more per row); with the cosine routing the dense product too.
        by = 2 * Hkv * d * e * (rows + kept) + B * Hq * case["w"] * d * e + 4 * Hkv * kept + 4 * B
        fl = 2.0 * Hq * case["w"] * d * rows + 6.0 * Hkv * d * rows
        if case["cosine"]:
            fl += sum(2.0 * Hkv * d * (n - int(case["rho"] * n)) * int(case["rho"] * n) for n in lens)
        return dict(bytes=by, flops=fl)
    L, T = case["layers"], case["steps"]
    rows = L * T * (sum(_lengths(case, 0, case["m"])) + B * (T + 1) // 2)
    # each token reads its layers' rows and one bias row for all heads
    by = rows * (2 * Hkv * d * e + (4 if case["bias"] else 0)) + L * T * B * d * e * (2 * Hq + 4 * Hkv)
    return dict(bytes=by, flops=4.0 * Hq * d * rows)


def tolerance(case):
    """About four times the distance of the library's results from the 64-bit ones: merged bf16
    values 4e-4 (rounding of the merged rows alone), turned keys, cosine-routed values and decoded
    rows 1.7e-3 (rounding of every element, and of the decode's weights), fp32 1.5e-7 with another
    order of the sums on top.  A single bf16 value may round the other way (2^-8 of it)."""
    if case["dtype"] == "fp32":
        return {"rel": 1e-5, "max": 1e-3}
    if case["kind"] == "decode":
        return {"rel": 7e-3, "max": 0.05}
    return {"rel": 7e-3 if case["rope"] or case["cosine"] else 2e-3, "max": 0.03}


# ---- the same in 64 bits ---------------------------------------------------------------------
_UNSURE = 1e-6  # two scores this close (relative) may be ordered either way in 32 bits


class _Ambiguous(Exception):
    pass


def _sure_top(x, k):
    """Mask of the k largest of x, ties to the lower index, and the relative gap at the cut."""
    v, i = torch.sort(x, descending=True, stable=True)
    mask = torch.zeros(x.shape[0], dtype=torch.bool, device=x.device)
    mask[i[:k]] = True
    gap = float((v[k - 1] - v[k]) / v[k - 1].clamp_min(1e-300)) if 0 < k < x.shape[0] else 1.0
    return mask, gap, (i[max(0, k - 1):k + 1] if 0 < k < x.shape[0] else i[:0])


def _exact_attention(Q, K, n, G, W):
    """a [Hkv][n]: causal softmax of the window's rows, summed over rows, mean over the group."""
    Hkv, d = K.shape[0], K.shape[-1]
    vis = torch.arange(n, device="cuda")[None, :] <= (n - W + torch.arange(W, device="cuda"))[:, None]
    a = torch.zeros((Hkv, n), dtype=torch.float64, device="cuda")
    for h in range(Hkv * G):
        s = Q[h].double() @ K[h // G, :n].double().T / math.sqrt(d)
        a[h // G] += torch.softmax(s.masked_fill(~vis, -math.inf), 1).sum(0)
    return a / G


def _exact_select(score, ncand, n, ms, per_head):
    """Kept masks [Hkv][n]."""
    Hkv = score.shape[0]
    tops = [_sure_top(score[h, :ncand], ms) for h in range(Hkv)]
    kept = torch.ones((Hkv, n), dtype=torch.bool, device="cuda")
    if per_head:
        if min(t[1] for t in tops) < _UNSURE:
            raise _Ambiguous
        kept[:, :ncand] = torch.stack([t[0] for t in tops])
        return kept
    votes = torch.stack([t[0] for t in tops]).sum(0)
    mean = score[:, :ncand].mean(0)
    members = torch.nonzero(votes > 0)[:, 0]
    chosen = votes > 0
    if members.numel() > ms:
        keep, gap, _ = _sure_top(mean[members], ms)
        if gap < _UNSURE:
            raise _Ambiguous
        chosen = torch.zeros_like(chosen)
        chosen[members[keep]] = True
    least = mean[chosen].min() if ms > 0 else mean.max()
    for mask, gap, edge in tops:
        # a head's own cut matters where no other head holds the token and the trim would keep it
        if gap < _UNSURE and bool(((votes[edge] <= mask[edge].long()) & (mean[edge] >= least * (1 - _UNSURE))).any()):
            raise _Ambiguous
    kept[:, :ncand] = chosen
    return kept


def _exact_bucket_targets(a, kept, n):
    """Merge target of every position [n] of one KV head (itself meaningless for kept ones)."""
    nb = (n + _BUCKET - 1) // _BUCKET
    pad = nb * _BUCKET - n
    ak = torch.nn.functional.pad(torch.where(kept, a, -1.0), (0, pad), value=-1.0).view(nb, _BUCKET)
    best, arg = ak.max(1)
    arg = (ak == best[:, None]).int().argmax(1)
    tau = torch.arange(nb, device="cuda") * _BUCKET + arg
    full = best >= 0
    at = torch.arange(nb, device="cuda")
    left = torch.where(full, at, -1).cummax(0).values
    right = torch.where(full, at, nb).flip(0).cummin(0).values.flip(0)
    dl = torch.where(left >= 0, at - left, nb + 1)
    dr = torch.where(right < nb, right - at, nb + 1)
    li, ri = left.clamp_min(0), right.clamp_max(nb - 1)
    take_left = (dl < dr) | ((dl == dr) & (best[li] >= best[ri]))
    home = torch.where(full, at, torch.where(take_left, li, ri))
    return tau[home][torch.arange(n, device="cuda") // _BUCKET]


def _exact_cosine_targets(V, kept):
    ki = torch.nonzero(kept)[:, 0]
    unit = V[ki] / V[ki].norm(dim=1, keepdim=True)
    target = torch.zeros(V.shape[0], dtype=torch.long, device="cuda")
    for j0 in range(0, V.shape[0], 4096):
        target[j0:j0 + 4096] = ki[(V[j0:j0 + 4096] @ unit.T).argmax(1)]
    return target


def _exact_rope(k, pos):
    """Each key turned back by (position - slot), half layout."""
    d = k.shape[-1]
    e = (pos - torch.arange(pos.shape[0], device="cuda")).double()
    w = _THETA ** (-2.0 * torch.arange(d // 2, device="cuda").double() / d)
    c, s = torch.cos(e[:, None] * w), torch.sin(e[:, None] * w)
    x, y = k[:, :d // 2], k[:, d // 2:]
    return torch.cat([x * c + y * s, y * c - x * s], 1)


def _exact_compress(case, seed):
    K, V, Q, lens = _compress_inputs(case, seed)
    B, Hq, Hkv, d, W = (case[k] for k in ("batch", "hq", "hkv", "d", "w"))
    G = Hq // Hkv
    cap = api.capacity(case["n"], case["rho"])
    Kc = torch.zeros((B, Hkv, cap, d), dtype=torch.float64, device="cuda")
    Vc = torch.zeros_like(Kc)
    bias = torch.zeros((B, Hkv, cap), dtype=torch.float64, device="cuda")
    for b, n in enumerate(lens):
        m = int(math.floor(case["rho"] * n))
        ms, ncand = m - _RECENT, n - _RECENT
        a = _exact_attention(Q[b], K[b], n, G, W)
        norm = torch.stack([V[b, h, :n].double().norm(dim=1) for h in range(Hkv)])
        c = torch.nn.functional.pad((a * norm)[:, :ncand], (_POOL // 2, _POOL // 2))
        score = sum(c[:, t:t + ncand] for t in range(_POOL)) / _POOL
        kept = _exact_select(score, ncand, n, ms, case["per_head"])
        R = torch.ones((Hkv, m), dtype=torch.float64, device="cuda")
        for h in range(Hkv):
            v = V[b, h, :n].double()
            pos = torch.nonzero(kept[h])[:, 0]
            slot = torch.cumsum(kept[h].long(), 0) - 1
            target = _exact_cosine_targets(v, kept[h]) if case["cosine"] else _exact_bucket_targets(a[h], kept[h], n)
            ev = torch.nonzero(~kept[h])[:, 0]
            t = target[ev]
            gate = ((v[ev] * v[t]).sum(1) / (norm[h, ev] * norm[h, t])).clamp(0.0, 1.0)
            w = gate * a[h, ev]
            num = a[h, pos, None] * v[pos]
            den = a[h, pos].clone()
            num.index_add_(0, slot[t], w[:, None] * v[ev])
            den.index_add_(0, slot[t], w)
            Vc[b, h, :m] = num / den[:, None]
            R[h] = den / a[h, pos]
            k = K[b, h, pos].double()
            Kc[b, h, :m] = _exact_rope(k, pos) if case["rope"] else k
        bias[b, :, :m] = _ALPHA * torch.log(R if case["per_head"] else R.mean(0, keepdim=True))
    return dict(K_c=Kc, V_c=Vc, bias=bias, lengths=torch.tensor([int(math.floor(case["rho"] * n)) for n in lens],
                                                                dtype=torch.int32, device="cuda"))


def _exact_decode(case, seed):
    K, V, bias, base, q, kn, vn, cap = _decode_inputs(case, seed)
    L, T, B, Hkv, d = case["layers"], case["steps"], case["batch"], case["hkv"], case["d"]
    lens = _lengths(case, seed, case["m"])
    out = torch.zeros(q.shape, dtype=torch.float64, device="cuda")
    for i in range(L):
        for b, n in enumerate(lens):
            for t in range(T):
                K[i, b, :, n + t], V[i, b, :, n + t] = kn[t, i, b], vn[t, i, b]
                if case["bias"]:
                    bias[i, b, :, n + t] = 0.0
                rows = n + t + 1
                s = q[t, i, b].double().view(Hkv, -1, d) @ K[i, b, :, :rows].double().transpose(1, 2) / math.sqrt(d)
                if case["bias"]:
                    s = s + bias[i, b, :, None, :rows].double()
                out[t, i, b] = (torch.softmax(s, 2) @ V[i, b, :, :rows].double()).view(-1, d)
    return dict(out=out, lengths=base + (torch.arange(base.shape[1], device="cuda") < B).int() * T,
                K=None, V=None, bias=None)


def exact(case, seed):
    if case["kind"] == "decode":
        return _exact_decode(case, seed)
    try:
        return _exact_compress(case, seed)
    except _Ambiguous:
        return None  # the kept set itself hangs on the last bits
