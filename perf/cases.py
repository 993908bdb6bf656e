"""The work this framework is measured on.

A case is one call a user makes: the bottleneck's forward, its backward, both
(a training step), the decoder alone (codes that a program has edited), the
standardisation update, the autograd layer, or the model around it. The
ranges: 1 to 65536 tokens, widths 64 to 2048, bf16 and fp32 rows, global
selection over 2^12 to 2^22 features (beams 4 to 16, codes of 8 to 128
entries) and the paper's per-level layouts, with and without tables.

``exact`` restates the method in 64 bits with torch alone: the field, the
seed matrix and the generators are built here from their definitions.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_20652_gb300 import dpb
from paper_2607_20652_gb300.layer import DPBLayer
from paper_2607_20652_gb300.transformer import ParityTransformer

WIDE = dict(d=768, m_bits=20, levels=5, beam=8, k=64, dtype="bf16")
GPT2 = dict(d=768, m_bits=16, levels=4, beam=8, k=32, dtype="bf16")
TINY = dict(d=64, m_bits=12, levels=3, beam=4, k=8, dtype="f32")
# the paper's per-level layouts: bits, children per parent, kept per level
LAYOUTS = {
    "small3l": dict(d=1024, bits=(10, 15, 17), keep=(16, 32, 64)),
    "small2l": dict(d=1024, bits=(10, 15), keep=(16, 32)),
    "large2l": dict(d=2048, bits=(11, 15), keep=(16, 32)),
}
ALPHA = 1e-4  # EMA rate: small enough that thousands of passes over one batch leave the tables sane


def listed():
    return [
        # the smallest workload: 256 fp32 tokens of 64 coordinates; launches and latency count
        dict(name="tiny_step", op="step", T=256, inputs="gaussian", **TINY),
        # a serving batch of 16 tokens through the wide dictionary
        dict(name="serve_forward", op="forward", T=16, inputs="planted", **WIDE),
        # fp32 rows at GPT-2 width: evaluation in full precision, a ragged batch
        dict(name="f32_forward", op="forward", T=3001, inputs="outliers", **{**GPT2, "dtype": "f32"}),
        # the autograd layer of a model of GPT-2 width, forward and backward: 8 x 1024 tokens with outlier rows
        dict(name="gpt2_layer", op="layer", T=8192, inputs="outliers", **GPT2),
        # the wide workload, its two directions apart
        dict(name="wide_forward", op="forward", T=65536, inputs="planted", **WIDE),
        dict(name="wide_backward", op="backward", T=65536, inputs="codes", **WIDE),
        # the far corner of the feature / code / beam sweep, forward and backward
        dict(name="sweep_step", op="step", T=32768, inputs="gaussian",
             **{**WIDE, "m_bits": 22, "beam": 16, "k": 128}),
        # codes edited by a program and decoded again, with no kept r; an odd batch
        dict(name="decode_edited", op="decode", T=20011, inputs="codes", **WIDE),
        # a training step with live standardisation: forward and backward with tables, then the EMA update
        dict(name="standardised_step", op="stats", T=8192, inputs="outliers", **WIDE),
        # the paper's three-level layout, forward and backward
        dict(name="paper3l_step", op="step", T=16384, layout="small3l", inputs="gaussian", dtype="bf16"),
        # the paper's wide two-level layout with tables (d = 2048), a ragged batch
        dict(name="paper2l_large_std", op="std_forward", T=4099, layout="large2l", inputs="gaussian", dtype="bf16"),
        # one block of the GPT-2-shape model: logits of 4 x 512 tokens (one block: each further one selects
        # again, and a selection turns last-bit differences into other codes)
        dict(name="model_logits", op="model", T=2048, inputs="tokens", **WIDE),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["global", "global", "global", "f32", "per_level", "layer", "stats"])
    if kind == "f32":
        d = rng.choice([64, 100, 256, 768])
        return dict(op=rng.choice(["forward", "step"]), T=_log_int(rng, 16, 3000), inputs="outliers", d=d,
                    m_bits=rng.choice([12, 14, 16]) if d <= 256 else 16, levels=rng.choice([3, 4]),
                    beam=rng.choice([4, 8]), k=rng.choice([8, 16, 32]), dtype="f32")
    if kind == "per_level":
        std = rng.random() < 0.3
        return dict(op="std_forward" if std else rng.choice(["forward", "step", "backward", "decode"]),
                    T=_log_int(rng, 8, 4096 if std else 16384), layout=rng.choice(sorted(LAYOUTS)),
                    inputs="gaussian", dtype="bf16")
    if kind in ("layer", "stats"):
        return dict(op=kind, T=_log_int(rng, 64, 16384), inputs="outliers", **WIDE)
    beam, k = rng.choice([4, 8, 16]), rng.choice([16, 32, 64, 128])
    op = rng.choice(["forward", "step", "backward", "decode"])
    return dict(op=op, T=_log_int(rng, 1, 32768 if beam > 8 or k > 64 else 65536),
                inputs=rng.choice(["gaussian", "outliers", "planted"]) if op in ("forward", "step") else "codes",
                d=rng.choice([512, 768, 768, 1024]), m_bits=rng.choice([16, 18, 20, 22]),
                levels=rng.choice([4, 5]), beam=beam, k=k, dtype="bf16")


# ---- the dictionary, from its definitions ------------------------------------------


def _poly(t):
    """p(z) of GF(2^t): the paper's for t = 10 and 11, else the smallest irreducible trinomial or pentanomial."""
    if t in (10, 11):
        return {10: (1 << 10) | 9, 11: (1 << 11) | 5}[t]

    def irreducible(p):
        for q in range(2, 1 << (t // 2 + 1)):
            a, n = p, q.bit_length()
            while a.bit_length() >= n:
                a ^= q << (a.bit_length() - n)
            if a == 0:
                return False
        return True

    top = 1 << t
    for a in range(1, t):
        if irreducible(top | (1 << a) | 1):
            return top | (1 << a) | 1
    found = [top | (1 << a) | (1 << b) | (1 << c) | 1 for a in range(3, t) for b in range(2, a) for c in range(1, b)]
    return next(p for p in sorted(found) if irreducible(p))


class _Dictionary:
    """Level bits, generators and the sign bits of a case's feature hierarchy (generator seed 0)."""

    def __init__(self, case, dev):
        lay = LAYOUTS.get(case.get("layout"))
        self.per_level = lay is not None
        self.d = lay["d"] if lay else case["d"]
        r0 = (self.d - 1).bit_length()
        if lay:
            self.bits, self.keep = list(lay["bits"]), list(lay["keep"])
            self.children = [0] + [256] * (len(self.bits) - 1)
            self.code_len = sum(self.keep)
        else:
            n, levels = case["m_bits"], case["levels"]
            self.bits = [r0 + (i * (n - r0)) // (levels - 1) for i in range(levels)]
            self.keep, self.children = [case["beam"]] * levels, [0] + [16] * (levels - 1)
            self.code_len = case["k"]
        self.levels, self.n_bits = len(self.bits), self.bits[-1]
        t = max(r0, (self.n_bits + 1) // 2)
        p = _poly(t)

        def mul(a, b):
            r = 0
            while b:
                r ^= a if b & 1 else 0
                b >>= 1
                a <<= 1
                a ^= p if a >> t else 0
            return r

        def powers(g):
            out = [1]
            while True:
                v = mul(out[-1], g)
                if v == 1:
                    return out
                out.append(v)

        exp = next(e for e in (powers(g) for g in range(2, 1 << t)) if len(e) == (1 << t) - 1)
        log = {v: i for i, v in enumerate(exp)}
        inv = [0] + [exp[-log[i] % len(exp)] for i in range(1, self.d)]
        rows = torch.tensor([i | (inv[i] << t) for i in range(self.d)], dtype=torch.int64)
        self.shifts = torch.arange(2 * t, device=dev)
        self.mbits = ((rows.to(dev)[:, None] >> self.shifts) & 1).float()  # [d, 2t]
        self.gens = [None]
        for lev in range(1, self.levels):
            s, got, mask = (lev * 0x9E3779B97F4A7C15) & (2**64 - 1), [], 2**64 - 1
            while len(got) < self.children[lev]:
                s = (s + 0x9E3779B97F4A7C15) & mask
                z = ((s ^ (s >> 30)) * 0xBF58476D1CE4E5B9) & mask
                z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
                g = (z ^ (z >> 31)) >> (64 - self.bits[lev])
                if g >> self.bits[lev - 1] and g not in got:
                    got.append(g)
            self.gens.append(torch.tensor(got, dtype=torch.int64, device=dev))

    def signs(self, c, dtype):
        """(-1)^parity(M AND c), [..., d], of feature indices c."""
        par = ((c[..., None] >> self.shifts) & 1).float() @ self.mbits.T
        return (1 - 2 * par.remainder_(2)).to(dtype)

    def synth(self, idx, coef):
        """sum_e coef_e phi_{idx_e}: [T, d] in coef's type, a few tokens at a time."""
        out = torch.zeros((len(idx), self.d), dtype=coef.dtype, device=coef.device)
        step = max(1, (1 << 26) // (idx.shape[1] * self.d))
        for a in range(0, len(idx), step):
            i, v = idx[a:a + step].long(), coef[a:a + step]
            hashed = i >= self.d
            o = torch.einsum("tk,tkd->td", torch.where(hashed, v, 0 * v), self.signs(i, v.dtype)) / math.sqrt(self.d)
            out[a:a + step] = o.scatter_add_(1, torch.where(hashed, 0 * i, i), torch.where(hashed, 0 * v, v))
        return out

    def analyse(self, idx, h):
        """<phi_{idx_e}, h>: [T, k]."""
        out = torch.empty(idx.shape, dtype=h.dtype, device=h.device)
        step = max(1, (1 << 26) // (idx.shape[1] * self.d))
        for a in range(0, len(idx), step):
            i, v = idx[a:a + step].long(), h[a:a + step]
            o = torch.einsum("td,tkd->tk", v, self.signs(i, v.dtype)) / math.sqrt(self.d)
            out[a:a + step] = torch.where(i < self.d, v.gather(1, i.clamp(max=self.d - 1)), o)
        return out

    def search(self, x, mu, sigma):
        """The encoder: (idx, z) of the code, and per level the raw scores of the distinct children considered."""
        dev, T = x.device, len(x)

        def z_of(s, c):
            return s if mu is None else (s - mu[c]) / sigma[c]

        def best(c, z, n):  # (|z| descending, index ascending), c ascending on entry
            o = torch.sort(z.abs(), dim=1, descending=True, stable=True).indices[:, :n]
            return c.gather(1, o), z.gather(1, o)

        c = torch.arange(self.d, device=dev).expand(T, -1)
        z = z_of(x, c)
        cands, considered = [(c, z)], []
        kept = [best(c, z, self.keep[0])]
        for lev in range(1, self.levels):
            gam = self.signs(self.gens[lev], x.dtype)
            par = kept[-1][0]
            c = (par[:, :, None] ^ self.gens[lev]).reshape(T, -1)
            s = ((self.signs(par, x.dtype) * x[:, None, :]) @ gam.T).reshape(T, -1) / math.sqrt(self.d)
            c, o = torch.sort(c, dim=1, stable=True)
            s = s.gather(1, o)
            new = torch.ones_like(c, dtype=torch.bool)
            new[:, 1:] = c[:, 1:] != c[:, :-1]
            z = torch.where(new, z_of(s, c), 0 * s)
            considered.append((c[new], s[new]))
            cands.append((c, z))
            kept.append(best(c, z, self.keep[lev]))
        if self.per_level:
            return torch.cat([k[0] for k in kept], 1), torch.cat([k[1] for k in kept], 1), considered
        return (*best(torch.cat([k[0] for k in cands], 1), torch.cat([k[1] for k in cands], 1), self.code_len),
                considered)


# ---- inputs -----------------------------------------------------------------------


def _planted(dic, T, g, dev):
    """A tree of planted features per token: 8 roots, then children of planted nodes, coefficients +-U[1, 2]."""
    per = [8] * (dic.levels - 1) + [32]
    idx = [torch.rand((T, dic.d), generator=g, device=dev).topk(8, dim=1).indices]
    for lev in range(1, dic.levels):
        pick = torch.rand((T, per[lev - 1] * 16), generator=g, device=dev).topk(per[lev], dim=1).indices
        idx.append(idx[-1].gather(1, pick // 16) ^ dic.gens[lev][pick % 16])
    idx = torch.cat(idx, 1)
    coef = (1 + torch.rand(idx.shape, generator=g, device=dev)) * \
        torch.randint(0, 2, idx.shape, generator=g, device=dev).mul(2).sub(1)
    x = dic.synth(idx, coef)
    return x + 0.1 * torch.randn(x.shape, generator=g, device=dev)


def _codes(dic, T, g, dev):
    """Codes as the encoder emits them: a fifth to three fifths basis entries, distinct, largest first."""
    k, lo, hi = dic.code_len, 1 << dic.bits[0], 1 << dic.n_bits
    nb = (k * (0.2 + 0.4 * torch.rand((T, 1), generator=g, device=dev))).long()
    basis = torch.rand((T, dic.d), generator=g, device=dev).topk(k, dim=1).indices
    step = torch.randint(1, (hi - lo) // k, (T, 1), generator=g, device=dev)
    start = torch.randint(0, hi - lo, (T, 1), generator=g, device=dev)
    j = torch.arange(k, device=dev)
    idx = torch.where(j < nb, basis, lo + (start + j * step) % (hi - lo))
    idx = idx.gather(1, torch.rand((T, k), generator=g, device=dev).argsort(1))
    val = torch.randn((T, k), generator=g, device=dev)
    return idx.int().contiguous(), val.gather(1, val.abs().argsort(1, descending=True)).contiguous()


def _inputs(case, seed, dev):
    """Everything drawn for a case, from the seed alone."""
    g = torch.Generator(dev).manual_seed(seed)
    dic = _Dictionary(case, dev)
    T, dt = case["T"], torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    s = {"dic": dic, "g": g}
    if case["inputs"] == "planted":
        x = _planted(dic, T, g, dev)
    else:
        x = torch.randn((T, dic.d), generator=g, device=dev)
        if case["inputs"] == "outliers":  # one row in twenty scaled by ten
            x = torch.where(torch.rand((T, 1), generator=g, device=dev) < 0.05, 10 * x, x)
    s["x"] = x.to(dt)
    if case["op"] in ("step", "backward", "stats", "layer"):
        s["gy"] = torch.randn((T, dic.d), generator=g, device=dev).to(dt)
    if case["op"] in ("backward", "decode"):
        s["idx"], s["val"] = _codes(dic, T, g, dev)
        s["r"] = dic.synth(s["idx"], s["val"])
        s["xnorm"] = s["x"].float().norm(dim=1)
    if case["op"] in ("stats", "std_forward"):
        m = 1 << dic.n_bits
        s["mu"] = 0.1 * torch.randn(m, generator=g, device=dev)
        s["sigma"] = 0.8 + 0.4 * torch.rand(m, generator=g, device=dev)
        s["sample"] = torch.randperm(T, generator=g, device=dev)[:64].int()
    return s


def _plan_args(case):
    if "layout" in case:
        lay = LAYOUTS[case["layout"]]
        n = len(lay["bits"])
        return dict(d=lay["d"], levels=n, bits=list(lay["bits"]), children=[0] + [256] * (n - 1),
                    k_per_level=list(lay["keep"]), select_mode=dpb.SELECT_PER_LEVEL, dtype="bf16")
    return dict(children=16, **{k: case[k] for k in ("d", "m_bits", "levels", "beam", "k", "dtype")})


def prepare(case, seed):
    dev = torch.device("cuda")
    if case["op"] == "model":
        torch.manual_seed(seed)
        kw = _plan_args(case)
        model = ParityTransformer(layers=1, d=kw.pop("d"), context=512, dpb=kw, device=dev).eval()
        return {"op": "model", "model": model, "ids": torch.randint(0, 50257, (case["T"] // 512, 512), device=dev)}
    s = _inputs(case, seed, dev)
    del s["g"], s["dic"]
    if case["op"] == "layer":
        return {**s, "op": "layer", "layer": DPBLayer(device=dev, **_plan_args(case)),
                "x": s["x"].requires_grad_(True)}
    return {**s, "op": case["op"], "plan": dpb.Plan(**_plan_args(case))}


def run(s):
    op = s["op"]
    if op == "model":
        with torch.no_grad():
            return s["model"](s["ids"])
    x = s["x"]
    if op == "layer":
        y = s["layer"](x)
        return {"y": y, "grad_x": torch.autograd.grad(y, x, s["gy"])[0]}
    plan = s["plan"]
    if op == "decode":
        return dpb.decode(plan, s["idx"], s["val"], s["xnorm"])
    if op == "backward":
        return dpb.backward(plan, x, s["idx"], s["val"], s["gy"], r=s["r"])
    mu, sigma = s.get("mu"), s.get("sigma")
    r = torch.empty(x.shape, dtype=torch.float32, device=x.device) if "gy" in s else None
    out = dpb.forward(plan, x, mu, sigma, r_out=r)
    if "gy" in s:
        out += dpb.backward(plan, x, out[0], out[1], s["gy"], sigma=sigma, r=r)
    if op == "stats":
        out += dpb.stats_step(plan, x, mu, sigma, ALPHA, s["sample"])
    return out


def work(case):
    T, b = case["T"], 4 if case["dtype"] == "f32" else 2
    if case["op"] == "model":  # the block's matrices, attention and the tied head
        d, v, s = 768, 50257, 512
        p = 4 * d * d + 2 * d * 3072 + v * d
        enc = (case["levels"] - 1) * case["beam"] * 16 * d
        return {"bytes": 2 * p + 8 * T + 2 * T * v, "flops": T * (2 * p + 2 * s * d + 2 * enc + 2 * case["k"] * d)}
    lay = LAYOUTS.get(case.get("layout"))
    d = lay["d"] if lay else case["d"]
    if lay:
        k, score = sum(lay["keep"]), sum(n * 256 * d for n in lay["keep"][:-1])
    else:
        k, score = case["k"], (case["levels"] - 1) * case["beam"] * 16 * d
    code, row = 8 * k, b * d
    fwd = {"bytes": 2 * row + code + 4, "flops": 2 * score + 2 * k * d}
    bwd = {"bytes": 3 * row + code + 4 * d + 4 * k, "flops": 4 * k * d}
    dec = {"bytes": code + 4 + row, "flops": 2 * k * d}
    w = {"forward": [fwd], "std_forward": [fwd], "decode": [dec], "backward": [bwd],
         "layer": [dict(bytes=4 * row, flops=fwd["flops"] + bwd["flops"])]}.get(case["op"])
    if w is None:  # a step reads x once and keeps its code and r on the way
        w = [fwd, dict(bytes=2 * row + 4 * k, flops=bwd["flops"])]
    total = {n: T * sum(p[n] for p in w) for n in ("bytes", "flops")}
    if case["op"] in ("std_forward", "stats"):
        total["bytes"] += 8 << (lay["bits"][-1] if lay else case["m_bits"])
    return total


# ---- 64-bit results ------------------------------------------------------------------


def exact(case, seed):
    if case["op"] == "model":
        return None
    s = _inputs(case, seed, torch.device("cuda"))
    dic, op, outs = s["dic"], case["op"], []
    tables = [s[n].double() if n in s else None for n in ("mu", "sigma")]
    step = 2048 if dic.per_level else 16384
    for a in range(0, case["T"], step):
        part = {n: v[a:a + step].double() for n, v in s.items() if n in ("x", "gy", "r", "val", "xnorm")}
        outs.append(_exact_rows(dic, op, part, s["idx"][a:a + step] if "idx" in s else None, *tables))
    cat = [None if o[0] is None else torch.cat(o) for o in zip(*outs)]
    if op == "layer":
        return {"y": cat[3], "grad_x": cat[4]}
    if op == "decode":
        return cat[0]
    if op == "stats":
        cat += _exact_moments(dic, s["x"].double(), s["sample"].long(), *tables)
    return tuple(cat)


def _exact_rows(dic, op, s, idx, mu, sigma):
    x = s["x"]
    nx = x.norm(dim=1, keepdim=True)
    head = []
    if idx is None:
        idx, val, _ = dic.search(x, mu, sigma)
        head = [None, val, nx[:, 0]]
        r = dic.synth(idx, val)
    else:
        val = s["val"]
        r = s["r"] if op == "backward" else dic.synth(idx, val)
    nr = r.norm(dim=1, keepdim=True)
    if op != "backward":
        head.append(r * (s["xnorm"][:, None] if op == "decode" else nx) / nr)
    if "gy" not in s:
        return head
    gr = (s["gy"] * r).sum(1, keepdim=True)
    gval = dic.analyse(idx, (nx / nr) * (s["gy"] - gr / nr**2 * r))
    coef = gval if sigma is None else gval / sigma[idx]
    return head + [dic.synth(idx, coef) + gr / nr * x / nx, gval]


def _exact_moments(dic, x, sample, mu, sigma):
    m = 1 << dic.n_bits
    n, s1, s2 = (torch.zeros(m, dtype=torch.float64, device=x.device) for _ in range(3))
    n[:dic.d], s1[:dic.d], s2[:dic.d] = len(x), x.sum(0), x.square().sum(0)
    for c, s in dic.search(x[sample], mu, sigma)[2]:
        n.index_add_(0, c, torch.ones_like(s))
        s1.index_add_(0, c, s)
        s2.index_add_(0, c, s * s)
    mean = s1 / n.clamp(min=1)
    dev = (s2 / n.clamp(min=1) - mean.square()).clamp(min=0).sqrt()
    return [torch.where(n >= 1, mu + ALPHA * (mean - mu), mu),
            torch.where(n >= 2, sigma + ALPHA * (dev - sigma), sigma)]
