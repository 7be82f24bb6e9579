"""What a user of the library has it do, as measurable cases: decode tokens, shard steps and prompt
prefills of the model shapes the repository works with (the 512-wide test layer, Llama-2-7B and 13B,
Llama-3-8B with grouped queries), through the calls of the ctypes binding.

A stack of a few layers stands for the whole model: every layer costs the same, and a few of them
exceed the L2 cache many times over, so each token streams its weights from device memory as the
32- or 40-layer model does.  Weights are N(0, 0.02^2), gains 1 + N(0, 0.02^2), embedding rows
N(0, 0.02^2) and cached keys and values N(0, (0.02 sqrt(d_model))^2), the spread their projections
have.

Kinds of case
  token        vt_embed and vt_decode_token for `tokens` token ids in turn, the cache growing by one each
  steps        one decode token through the per-device calls, as a program with one device per
               shard makes them: vt_decode_step of every shard, vt_combine, vt_kv_advance, captured
               once as a CUDA graph and replayed
  static       vt_decode_step_static of one device's attention shards
  prefill      vt_embed and vt_prefill_tokens of a prompt behind `kv_len` cached positions
  shardprefill vt_prefill of one device's shards of every layer with the combines in between
A pass ends by taking the cache lengths back to `kv_len`, as a program does that tries another
continuation, so that it can be repeated.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_07046_gb300 import vt

FAMILIES = {
    "tiny": dict(d_model=512, n_heads=8, n_kv_heads=8, d_head=64, d_ffn=1408, theta=1e4),
    "7b": dict(d_model=4096, n_heads=32, n_kv_heads=32, d_head=128, d_ffn=11008, theta=1e4),
    "13b": dict(d_model=5120, n_heads=40, n_kv_heads=40, d_head=128, d_ffn=13824, theta=1e4),
    "8b": dict(d_model=4096, n_heads=32, n_kv_heads=8, d_head=128, d_ffn=14336, theta=5e5),
}
EPS = 1e-5
VOCAB = 32000
NAMES = ("attn_norm", "wq", "wk", "wv", "wo", "ffn_norm", "w_gate", "w_up", "w_down")


def _case(name, kind, family, layers, heads, kv_len, rows=0, tokens=0, window=0, bits="16", comm=16, device=0, shift=0):
    """heads: query heads per device, as "8,8,8,8"; FFN columns are split in the same proportion.
    bits: weight bits of the shards, in turn over (layer, device, block).  shift: heads and columns
    that device 0 hands to device 1 in every odd layer (a per-layer partition)."""
    c = dict(kind=kind, family=family, layers=layers, heads=heads, kv_len=kv_len, rows=rows, tokens=tokens,
             window=window, bits=bits, comm=comm, device=device, shift=shift)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest model: launch and latency bound
        _case("tiny token", "token", "tiny", 1, "4,4", 128, tokens=4),
        # the ordinary decode token: four even devices, 1024 cached positions
        _case("7b token", "token", "7b", 4, "8,8,8,8", 1024, tokens=4),
        # uneven devices and a longer cache
        _case("13b token uneven", "token", "13b", 3, "20,12,8", 2048, tokens=2),
        # grouped queries at a long cache
        _case("8b token long", "token", "8b", 4, "8,8,8,8", 4096, tokens=2),
        # every device holds its shards at 8 bits
        _case("7b token int8", "token", "7b", 3, "8,8,8,8", 1024, tokens=2, bits="8"),
        # heterogeneous devices: 4-, 8- and 16-bit shards, ranges that differ by layer, 8-bit partials
        _case("8b token mixed", "token", "8b", 3, "12,8,12", 700, tokens=2, bits="4,4,8,4,16", comm=8, shift=4),
        # the per-device program of one token
        _case("7b shard steps", "steps", "7b", 2, "8,8,8,8", 1024),
        # the attention step of a caller that cannot allocate
        _case("8b static step", "static", "8b", 3, "8,8,8,8", 4096, device=1),
        # an ordinary prompt
        _case("7b prefill 512", "prefill", "7b", 2, "8,8,8,8", 0, rows=512),
        # the next short turn of a chat: odd length behind a cached history
        _case("8b prefill 77", "prefill", "8b", 2, "8,8,8,8", 300, rows=77),
        # a long document on uneven devices
        _case("13b prefill 2048", "prefill", "13b", 1, "20,12,8", 0, rows=2048),
        # one device's part of a prompt, sliding-window attention
        _case("8b shard prefill", "shardprefill", "8b", 2, "8,16,8", 700, rows=333, window=512, device=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cuts(rng, units, n):
    at = sorted(rng.sample(range(1, units), n - 1))
    return [b - a for a, b in zip([0] + at, at + [units])]


def draw(rng):
    kind = rng.choice(["token", "token", "token", "steps", "static", "prefill", "prefill", "shardprefill"])
    fam = rng.choice(["tiny", "7b", "13b", "8b", "8b"])
    f = FAMILIES[fam]
    group = f["n_heads"] // f["n_kv_heads"]
    n = rng.choice([1, 2, 3, 4])
    parts = _cuts(rng, f["n_kv_heads"], n) if rng.random() < 0.5 else [f["n_kv_heads"] // n] * (n - 1) + [
        f["n_kv_heads"] - (n - 1) * (f["n_kv_heads"] // n)]
    heads = ",".join(str(u * group) for u in parts)
    layers = 1 if fam == "13b" else 2
    window = rng.choice([0, 0, 0, _log(rng, 16, 2048)])
    device = rng.randrange(n)
    if kind in ("token", "steps", "static"):
        kv_len = _log(rng, 1, 6000) if rng.random() < 0.9 else 0
        if kind == "static":
            return _case(None, kind, fam, layers, heads, kv_len, window=window, device=device)
        if kind == "steps":
            return _case(None, kind, fam, layers, heads, kv_len, window=window)
        bits = rng.choice(["16", "16", "8", "4", "8,4,16"])
        comm = rng.choice([16, 16, 16, 8, 4])
        shift = group if n > 1 and parts[0] > 1 and rng.random() < 0.3 else 0
        return _case(None, kind, fam, layers, heads, kv_len, tokens=rng.choice([1, 2, 3]), window=window, bits=bits,
                     comm=comm, shift=shift)
    rows = _log(rng, 2, 2048 if fam == "tiny" else 900)
    kv_len = _log(rng, 1, 2000) if rng.random() < 0.5 else 0
    return _case(None, kind, fam, 1, heads, kv_len, rows=rows, window=window, device=device)


# ------------------------------------------------------------------ inputs, from the seed alone

def _ranges(case):
    """(head ranges per layer, FFN column ranges per layer)."""
    f = FAMILIES[case["family"]]
    heads = [int(x) for x in case["heads"].split(",")]
    H, F = f["n_heads"], f["d_ffn"]
    per_head = F / H
    lh, lc = [], []
    for l in range(case["layers"]):
        hs = list(heads)
        if case["shift"] and l % 2:
            hs[0] -= case["shift"]
            hs[1] += case["shift"]
        ends = np.cumsum([0] + hs)
        cols = [int(round(e * per_head)) for e in ends]
        lh.append([(int(a), int(b)) for a, b in zip(ends, ends[1:])])
        lc.append(list(zip(cols, cols[1:])))
    return lh, lc


def _normal(seed, index, shape, mean=0.0, std=1.0):
    g = torch.Generator(device="cuda").manual_seed((int(seed) * 4096 + index) % (1 << 62))
    return (torch.randn(shape, generator=g, device="cuda") * std + mean).half()


def _layer(case, seed, l):
    f = FAMILIES[case["family"]]
    D, F, q, k = f["d_model"], f["d_ffn"], f["n_heads"] * f["d_head"], f["n_kv_heads"] * f["d_head"]
    shapes = dict(attn_norm=(D,), wq=(q, D), wk=(k, D), wv=(k, D), wo=(D, q), ffn_norm=(D,), w_gate=(F, D),
                  w_up=(F, D), w_down=(D, F))
    return {n: _normal(seed, 16 * l + i, shapes[n], 1.0 if n.endswith("norm") else 0.0, 0.02)
            for i, n in enumerate(NAMES)}


def _cached(case, seed, l):
    """Cached keys and values of layer l, [KV heads, positions, head dim]."""
    f = FAMILIES[case["family"]]
    shape, std = (f["n_kv_heads"], case["kv_len"], f["d_head"]), 0.02 * math.sqrt(f["d_model"])
    return _normal(seed, 16 * l + 10, shape, 0.0, std), _normal(seed, 16 * l + 11, shape, 0.0, std)


def _embedding(case, seed):
    return _normal(seed, 4000, (VOCAB, FAMILIES[case["family"]]["d_model"]), 0.0, 0.02)


def _ids(case, seed, n):
    g = torch.Generator(device="cuda").manual_seed(int(seed) * 4096 + 4001)
    return torch.randint(0, VOCAB, (n,), generator=g, device="cuda", dtype=torch.int32)


def _hidden(case, seed, rows):
    return _normal(seed, 4002, (rows, FAMILIES[case["family"]]["d_model"]), 0.0, 0.5)


def _bits(case, l, d, block):
    b = case["bits"].split(",")
    return int(b[(l * 8 + d * 2 + block) % len(b)])


def _new_rows(case):
    return case["rows"] or case["tokens"] or 1


# ------------------------------------------------------------------ the user's program

class State:
    def __init__(self, case, seed):
        f = FAMILIES[case["family"]]
        self.case, self.layers, self.D = case, case["layers"], f["d_model"]
        self.lh, self.lc = _ranges(case)
        self.devices = len(self.lh[0])
        self.model = self.part = self.kv = 0
        kind, new = case["kind"], _new_rows(case)
        embeds = kind in ("token", "prefill")
        cap = case["kv_len"] + new + 8
        shapes = vt.make_shapes(self.layers, self.D, f["n_heads"], f["n_kv_heads"], f["d_head"], f["d_ffn"],
                                VOCAB if embeds else 0, cap, EPS, f["theta"])
        self.model = vt.vt_model_create(shapes)
        for l in range(self.layers):
            vt.vt_model_load_layer(self.model, l, {n: w.cpu().numpy() for n, w in _layer(case, seed, l).items()})
        if case["window"]:
            vt.vt_model_set_window(self.model, -1, case["window"])
        if case["shift"]:
            self.part = vt.vt_partition_create_layers(self.model, self.lh, self.lc)
        else:
            self.part = vt.vt_partition_create(self.model, self.lh[0], self.lc[0])
        for l in range(self.layers):
            for d in range(self.devices):
                for block in (vt.VT_BLOCK_ATTN, vt.VT_BLOCK_FFN):
                    if _bits(case, l, d, block) != 16:
                        vt.vt_partition_set_precision(self.part, (l, d, block), _bits(case, l, d, block))
        if case["comm"] != 16:
            vt.vt_partition_set_comm_bits(self.part, -1, case["comm"])
        self.kv = vt.vt_kv_create(self.part, cap)
        if case["kv_len"]:
            group = f["n_heads"] // f["n_kv_heads"]
            for l in range(self.layers):
                k, v = (t.cpu().numpy() for t in _cached(case, seed, l))
                for d, (a, b) in enumerate(self.lh[l]):
                    if b > a:
                        vt.vt_kv_write_raw(self.kv, l, d, k[a // group:b // group], v[a // group:b // group])
            vt.vt_kv_set_length(self.kv, -1, case["kv_len"])
        if embeds:
            vt.vt_model_load_embedding(self.model, _embedding(case, seed).cpu().numpy())
            self.ids = _ids(case, seed, new)
            self.x = torch.empty(new, self.D, dtype=torch.float16, device="cuda")
        else:
            self.x = _hidden(case, seed, new)
        n_part = self.devices if kind == "steps" else 1
        self.out = torch.empty(new, self.D, dtype=torch.float16, device="cuda")
        if not embeds:
            # fp32 partials of every layer's two blocks, and the hidden rows between them
            self.attn = torch.empty(self.layers, n_part, new, self.D, dtype=torch.float32, device="cuda")
            self.ffn = torch.empty_like(self.attn)
            self.h = torch.empty(self.layers, 2, new, self.D, dtype=torch.float16, device="cuda")
        self.graph = None
        if kind == "steps":
            self.one_token_of_steps()
            torch.cuda.synchronize()
            self.graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(self.graph):
                self.one_token_of_steps()

    def one_token_of_steps(self):
        cur = self.x
        for l in range(self.layers):
            for d in range(self.devices):
                vt.vt_decode_step(self.part, (l, d, vt.VT_BLOCK_ATTN), cur, self.kv, self.attn[l, d])
            vt.vt_combine(list(self.attn[l]), cur, self.h[l, 0], 1, self.D)
            for d in range(self.devices):
                vt.vt_decode_step(self.part, (l, d, vt.VT_BLOCK_FFN), self.h[l, 0], None, self.ffn[l, d])
            vt.vt_combine(list(self.ffn[l]), self.h[l, 0], self.h[l, 1], 1, self.D)
            cur = self.h[l, 1]
        vt.vt_kv_advance(self.kv, -1, 1)
        vt.vt_kv_advance(self.kv, -1, -1)

    def __del__(self):
        try:
            torch.cuda.synchronize()
            vt.vt_kv_destroy(self.kv)
            vt.vt_partition_destroy(self.part)
            vt.vt_model_destroy(self.model)
        except Exception:  # the interpreter is closing down
            pass


def prepare(case, seed):
    return State(case, seed)


def run(s):
    case, kind, dev = s.case, s.case["kind"], s.case["device"]
    if kind == "token":
        for t in range(case["tokens"]):
            vt.vt_embed(s.model, s.ids[t:t + 1], s.x[t:t + 1])
            vt.vt_decode_token(s.part, s.kv, s.x[t:t + 1], s.out[t:t + 1])
        vt.vt_kv_advance(s.kv, -1, -case["tokens"])
        return s.out
    if kind == "steps":
        s.graph.replay()
        return {"attn": s.attn, "ffn": s.ffn, "h": s.h}
    if kind == "static":
        for l in range(s.layers):
            vt.vt_decode_step_static(s.part, (l, dev, vt.VT_BLOCK_ATTN), s.x, s.kv, s.attn[l, 0])
        return s.attn
    if kind == "prefill":
        vt.vt_embed(s.model, s.ids, s.x)
        vt.vt_prefill_tokens(s.part, s.kv, s.x, case["rows"], s.out)
        vt.vt_kv_advance(s.kv, -1, -case["rows"])
        return s.out
    rows, cur = case["rows"], s.x
    for l in range(s.layers):
        vt.vt_prefill(s.part, (l, dev, vt.VT_BLOCK_ATTN), cur, rows, s.kv, s.attn[l, 0])
        vt.vt_combine([s.attn[l, 0]], cur, s.h[l, 0], rows, s.D)
        vt.vt_prefill(s.part, (l, dev, vt.VT_BLOCK_FFN), s.h[l, 0], rows, None, s.ffn[l, 0])
        vt.vt_combine([s.ffn[l, 0]], s.h[l, 0], s.h[l, 1], rows, s.D)
        cur = s.h[l, 1]
    return {"attn": s.attn, "ffn": s.ffn, "h": s.h}


# ------------------------------------------------------------------ work

def _attended(case, n_rows):
    """Sum over the new rows of the positions each attends to, and the cached positions read."""
    w, L = case["window"], case["kv_len"]
    total = sum(min(L + i + 1, w) if w else L + i + 1 for i in range(n_rows))
    old = min(L, w - 1) if w else L
    return total, old


def work(case):
    f = FAMILIES[case["family"]]
    D, dh = f["d_model"], f["d_head"]
    group = f["n_heads"] // f["n_kv_heads"]
    kind, new = case["kind"], _new_rows(case)
    lh, lc = _ranges(case)
    devs = [case["device"]] if kind in ("static", "shardprefill") else range(len(lh[0]))
    total, old = _attended(case, new)
    nbytes, flops = 0.0, 0.0
    # a token of the decode kinds streams the weights again: they exceed the caches
    passes, rows = (new, 1) if kind == "token" else (1, new)
    for l in range(case["layers"]):
        for d in devs:
            hq, c = lh[l][d][1] - lh[l][d][0], lc[l][d][1] - lc[l][d][0]
            hk = hq // group
            attn_w, ffn_w = (hq * 2 + hk * 2) * dh * D, 3 * D * c * (kind != "static")
            for block, w in ((0, attn_w), (1, ffn_w)):
                bits = _bits(case, l, d, block)
                per = 2.0 if bits == 16 else (1.0 if bits == 8 else 0.5) + 2 / 32
                nbytes += passes * w * per
                flops += 2.0 * w * new
            kv_read = (total if kind == "token" else old) * hk * dh * 4
            nbytes += kv_read + new * hk * dh * 4
            flops += 4.0 * hq * dh * total
            if kind in ("steps", "static", "shardprefill"):  # partials are results of these calls
                nbytes += rows * D * 4 * (1 if kind == "static" else 2)
    nbytes += new * D * 2 * (3 if kind in ("token", "prefill") else 1)
    if kind in ("steps", "shardprefill"):
        nbytes += case["layers"] * 2 * new * D * 2
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------ tolerance

def tolerance(case):
    """About four times what each path shows against exact().  The fp32 partials of a decode step
    differ by the order of their sums; hidden rows and cache entries are rounded to 16 bits once a
    block, a prefill's operands too; a partial sent at 8 or 4 bits moves by a whole step where a
    value lies at a tie."""
    kind, comm = case["kind"], case["comm"]
    if kind == "static":
        return {"rel": 4e-5, "max": 2e-4}
    if kind == "steps":
        return {"rel": 1.2e-3, "max": 8e-3}
    if kind == "token":
        return {16: {"rel": 2.5e-3, "max": 2e-2}, 8: {"rel": 1.8e-2, "max": 0.1}, 4: {"rel": 0.3, "max": 0.95}}[comm]
    return {"rel": 4e-3, "max": 3e-2}


# ------------------------------------------------------------------ the same in 64 bits

def _blocks(w, bits):
    """Values of weight rows [rows, k] (fp16 values in fp32) stored at `bits`: blocks of 32 along k."""
    if bits == 16:
        return w.double()
    qmax = 127.0 if bits == 8 else 7.0
    rows, k = w.shape
    pad = torch.zeros(rows, -k % 32, dtype=torch.float32, device=w.device)
    b = torch.cat([w.float(), pad], 1).view(rows, -1, 32)
    d = (b.abs().amax(2, keepdim=True) / qmax).half().float()
    q = torch.where(d > 0, (b / torch.where(d > 0, d, torch.ones_like(d))).round().clamp(-qmax, qmax), torch.zeros_like(b))
    return (q.double() * d.double()).view(rows, -1)[:, :k]


def _sent(p, bits):
    """A partial [rows, D] as it reaches the combine."""
    return p if bits == 16 else _blocks64(p, bits)


def _blocks64(p, bits):
    qmax = 127.0 if bits == 8 else 7.0
    b = p.view(p.shape[0], -1, 32)
    d = (b.abs().amax(2, keepdim=True) / qmax).half().double()
    q = torch.where(d > 0, (b / torch.where(d > 0, d, torch.ones_like(d))).round().clamp(-qmax, qmax), torch.zeros_like(b))
    return (q * d).reshape(p.shape)


def _norm(x, gain):
    return x * torch.rsqrt((x * x).mean(1, keepdim=True) + EPS) * gain.double()


def _rope(x, pos, theta):
    """x [rows, heads, dh], rotate-half."""
    half = x.shape[2] // 2
    freq = theta ** (-2.0 * torch.arange(half, device=x.device, dtype=torch.float64) / x.shape[2])
    ang = pos[:, None].double() * freq[None, :]
    c, s = ang.cos()[:, None, :], ang.sin()[:, None, :]
    a, b = x[..., :half], x[..., half:]
    return torch.cat([a * c - b * s, a * s + b * c], 2)


def _attn_partial(case, w, kc, vc, x, p0, h0, h1, bits):
    """fp64 attention partial of heads [h0, h1) for rows x at positions p0.., appending to kc / vc
    [KV heads, positions, dh] (16-bit values in fp64)."""
    f = FAMILIES[case["family"]]
    dh, group = f["d_head"], f["n_heads"] // f["n_kv_heads"]
    k0, k1, n = h0 // group, h1 // group, x.shape[0]
    xn = _norm(x, w["attn_norm"])
    pos = torch.arange(p0, p0 + n, device=x.device)
    proj = lambda name, a, b: (xn @ _blocks(w[name][a * dh:b * dh], bits).T).view(n, b - a, dh)  # noqa: E731
    q = _rope(proj("wq", h0, h1), pos, f["theta"])
    kc[k0:k1, p0:p0 + n] = _rope(proj("wk", k0, k1), pos, f["theta"]).half().double().transpose(0, 1)
    vc[k0:k1, p0:p0 + n] = proj("wv", k0, k1).half().double().transpose(0, 1)
    at = torch.arange(p0 + n, device=x.device)
    seen = at[None, :] <= pos[:, None]
    if case["window"]:
        seen &= at[None, :] > pos[:, None] - case["window"]
    out = torch.empty(n, h1 - h0, dh, dtype=torch.float64, device=x.device)
    for h in range(h1 - h0):
        kv = (h0 + h) // group
        s = (q[:, h] @ kc[kv, :p0 + n].T) / math.sqrt(dh)
        out[:, h] = torch.softmax(s.masked_fill(~seen, -math.inf), 1) @ vc[kv, :p0 + n]
    return out.reshape(n, -1) @ _blocks(w["wo"][:, h0 * dh:h1 * dh], bits).T


def _ffn_partial(w, x, c0, c1, bits):
    xn = _norm(x, w["ffn_norm"])
    g, u = xn @ _blocks(w["w_gate"][c0:c1], bits).T, xn @ _blocks(w["w_up"][c0:c1], bits).T
    return (g * torch.sigmoid(g) * u) @ _blocks(w["w_down"][:, c0:c1], bits).T


def exact(case, seed):
    f = FAMILIES[case["family"]]
    kind, new, L = case["kind"], _new_rows(case), case["kv_len"]
    lh, lc = _ranges(case)
    devs = [case["device"]] if kind in ("static", "shardprefill") else range(len(lh[0]))
    if kind in ("token", "prefill"):
        x = _embedding(case, seed)[_ids(case, seed, new).long()].double()
    else:
        x = _hidden(case, seed, new).double()
    attn, ffn, hid = [], [], []
    cur = x
    for l in range(case["layers"]):
        w = _layer(case, seed, l)
        kc = torch.zeros(f["n_kv_heads"], L + new, f["d_head"], dtype=torch.float64, device="cuda")
        vc = torch.zeros_like(kc)
        if L:
            k, v = _cached(case, seed, l)
            kc[:, :L], vc[:, :L] = k.double(), v.double()
        ap = [_attn_partial(case, w, kc, vc, cur, L, *lh[l][d], _bits(case, l, d, 0)) for d in devs]
        attn.append(torch.stack(ap))
        if kind == "static":
            continue
        h = (cur + sum(_sent(p, case["comm"]) for p in ap)).half().double()
        fp = [_ffn_partial(w, h, *lc[l][d], _bits(case, l, d, 1)) for d in devs]
        ffn.append(torch.stack(fp))
        nxt = h + sum(_sent(p, case["comm"]) for p in fp)
        hid.append(torch.stack([h, nxt.half().double()]))
        cur = nxt if l == case["layers"] - 1 else nxt.half().double()
    if kind == "static":
        return torch.stack(attn)
    if kind in ("token", "prefill"):
        return cur
    return {"attn": torch.stack(attn), "ffn": torch.stack(ffn), "h": torch.stack(hid)}
