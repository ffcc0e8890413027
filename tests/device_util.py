"""Attention calls on inputs made on the device, and their fp64 reference in plain
torch: for prefixes too long for the host generator and the oracle."""
import copy
import math

import torch

from tests.gpu_util import LSE_ABS

# The kernels round the softmax weights and the outputs to bf16 (relative error at
# most U = 2^-8) and normalise with the sum of the rounded weights, so that with
# weights w_j (1 + e_j)  out - o = sum w_j e_j (v_j - o) / sum w_j (1 + e_j):  at most
# U sum w_j |v_j - o|, which the weighted deviation of the values bounds.  A score off
# by d moves a weight by the factor e^d: d is below the lse's bound.
U = 2.0 ** -8
SUMS = 2.0 ** -21  # error of an fp32 sum of up to 128 products, of their magnitudes' sum
# The largest error of an element of a split query, of its row's largest element:
# two parts end at e4m3's smallest value 2^-9 (error 2^-10) with the largest element
# at 2^7 or above; three end at e5m2's 2^-16 with the largest above 2^14.
SPLIT = {2: 2.0 ** -17, 3: 2.0 ** -31}


class Call:
    """One layer's call: sequences of prefixes P and blocks T, H kv heads of G query
    heads, D wide; kf8 / vf8: prefix keys / values stored as e4m3.  What lies past the
    lengths is NaN.  sharp: deviation of a score (natural units) is about its value."""

    def __init__(self, P, T, G, H, D, kf8=False, vf8=False, capacity=None, seed=0, sharp=1.0):
        import paper_2609_34538_gb300 as das
        self.P, self.T, self.G, self.H, self.D = list(P), list(T), G, H, D
        self.kf8, self.vf8, self.f8 = kf8, vf8, kf8 or vf8
        self.split = SPLIT[2 if D == 128 and not vf8 else 3]
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        B, rows = len(P), max(T)
        cap = capacity or max(max(P), 1)
        normal = lambda *shape: torch.randn(shape, generator=g, device="cuda").to(torch.bfloat16)
        # two depths: depth 1 (e4m3 in a das_kv_cache_f8) and depth R = 2
        k, v = normal(B, cap, H, D), normal(B, cap, H, D)
        self.q = (normal(B, rows, H * G, D) * sharp).to(torch.bfloat16)
        self.kb, self.vb = normal(B, rows, H, D), normal(B, rows, H, D)
        for b, (p, t) in enumerate(zip(P, T)):
            k[b, p:], v[b, p:] = math.nan, math.nan
            self.q[b, t:], self.kb[b, t:], self.vb[b, t:] = math.nan, math.nan, math.nan
        self.kd, self.vd = (1 if kf8 else 2), (1 if vf8 else 2)
        if self.f8:
            low = lambda x: x.to(torch.float8_e4m3fn).view(torch.uint8)[None, None].contiguous()
            self.cache = das.DepthKVCacheF8(k[None], v[None], low(k), low(v))
            self.ws = das.new_workspace_f8(self.cache, H * G, rows)
        else:
            self.cache = das.DepthKVCache(k[None, None].repeat(2, 1, 1, 1, 1, 1),
                                          v[None, None].repeat(2, 1, 1, 1, 1, 1))
            self.ws = das.new_workspace(self.cache, H * G, rows)
        self.pl = torch.tensor(self.P, dtype=torch.int32, device="cuda")
        self.bl = torch.tensor(self.T, dtype=torch.int32, device="cuda")

    def with_capacity(self, cap):
        """The same call over a cache of that capacity."""
        import paper_2609_34538_gb300 as das
        c = copy.copy(self)
        k = self.cache.k_top[0] if self.f8 else self.cache.k[1, 0]
        grown = torch.full((len(self.P), cap) + k.shape[2:], math.nan, dtype=torch.bfloat16,
                           device="cuda")
        n = min(cap, k.shape[1])
        def fit(x):  # [..][B][capacity][H][D]
            y = grown if x.dtype == torch.bfloat16 else torch.full_like(grown, 0x7F, dtype=torch.uint8)
            y = y.expand(x.shape[:-4] + y.shape).clone()
            y[..., :n, :, :] = x[..., :n, :, :]
            return y
        if self.f8:
            c.cache = das.DepthKVCacheF8(*map(fit, (self.cache.k_top, self.cache.v_top,
                                                    self.cache.k_low, self.cache.v_low)))
            c.ws = das.new_workspace_f8(c.cache, self.H * self.G, self.q.shape[1])
        else:
            c.cache = das.DepthKVCache(fit(self.cache.k), fit(self.cache.v))
            c.ws = das.new_workspace(c.cache, self.H * self.G, self.q.shape[1])
        return c

    # the stored keys and values that the call reads, [B][cap][H][D] (views, to be edited)
    @property
    def k(self):
        if not self.f8:
            return self.cache.k[1, 0]
        return self.cache.k_low[0, 0].view(torch.float8_e4m3fn) if self.kf8 else self.cache.k_top[0]

    @property
    def v(self):
        if not self.f8:
            return self.cache.v[1, 0]
        return self.cache.v_low[0, 0].view(torch.float8_e4m3fn) if self.vf8 else self.cache.v_top[0]

    def run(self, scale=0.0, **kw):
        import paper_2609_34538_gb300 as das
        fn = das.das_mature_v_attention_f8 if self.f8 else das.das_mature_v_attention
        out, lse = fn(self.cache, 0, self.kd, self.vd, self.pl, self.bl, self.q, self.kb, self.vb,
                      self.ws, softmax_scale=scale, **kw)
        return out, lse

    def reference(self, scale=0.0):
        """(out, lse, bound of the outputs' errors, bound of the lse's) in fp64; rows past a
        block 0 and -inf."""
        H, G, D = self.H, self.G, self.D
        out, dev = (torch.zeros(self.q.shape, dtype=torch.float64, device="cuda") for _ in range(2))
        lse = torch.full((len(self.P), H * G, self.q.shape[1]), -math.inf, dtype=torch.float64,
                         device="cuda")
        for b, (p, t) in enumerate(zip(self.P, self.T)):
            if t == 0:
                continue
            K = torch.cat([self.k[b, :p].double(), self.kb[b, :t].double()]).permute(1, 0, 2)
            V = torch.cat([self.v[b, :p].double(), self.vb[b, :t].double()]).permute(1, 0, 2)
            Q = self.q[b, :t].double().reshape(t, H, G, D).permute(1, 2, 0, 3).reshape(H, G * t, D)
            s = Q @ K.transpose(1, 2) * (scale if scale > 0 else 1 / math.sqrt(D))
            i = torch.arange(t, device="cuda").repeat(G)
            s[:, :, p:].masked_fill_(torch.arange(t, device="cuda")[None] > i[:, None], -math.inf)
            l = torch.logsumexp(s, -1)
            w = torch.exp(s - l[..., None])
            o = w @ V
            rows = lambda x: x.reshape(H, G, t, D).permute(2, 0, 1, 3).reshape(t, H * G, D)
            out[b, :t], dev[b, :t] = rows(o), rows(w @ V.square() - o.square())
            lse[b, :, :t] = l.reshape(H * G, t)
        # a score's error (natural units): fp32 sums of the products, and the part of a
        # split query that is dropped times the keys
        off = torch.zeros(lse.shape, dtype=torch.float64, device="cuda")
        for b, (p, t) in enumerate(zip(self.P, self.T)):
            if t:
                K = torch.cat([self.k[b, :p].double(), self.kb[b, :t].double()])
                K = K.abs().permute(1, 2, 0)  # [H][D][keys]
                q = self.q[b, :t].double().abs().reshape(t, H, G, D).permute(1, 2, 0, 3)
                d = SUMS * (q.reshape(H, G * t, D) @ K).amax(-1)
                if self.kf8:
                    d = d + self.split * q.reshape(H, G * t, D).amax(-1) * K.sum(1).amax(-1)[:, None]
                off[b, :, :t] = d.reshape(H * G, t)
        off = LSE_ABS + off * (scale if scale > 0 else 1 / math.sqrt(D))
        w = 2 * off.permute(0, 2, 1)[..., None]
        return out, lse, 1.01 * ((U + w) * dev.clamp(min=0).sqrt() + U * out.abs()), off

    def status(self):
        import paper_2609_34538_gb300 as das
        return das.workspace_status(self.ws)


def assert_rows(out, lse, ref, keep=None):
    """Every row's outputs and lse within the reference's bounds; keep: the rows
    [B][T][Hq] compared."""
    err = ((out.double() - ref[0]).abs() - ref[2]).amax(-1)
    l, xl = lse.double().permute(0, 2, 1), ref[1].permute(0, 2, 1)
    le = torch.where(torch.isneginf(xl) & torch.isneginf(l), 0.0, (l - xl).abs()) - ref[3].permute(0, 2, 1)
    if keep is not None:
        err, le = err[keep], le[keep]
    assert bool((err <= 0).all()), f"outputs beyond their bound by {err.max().item():.3e}"
    assert bool((le <= 0).all()), f"lse beyond its bound by {le.max().item():.3e}"
