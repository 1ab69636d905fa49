"""The work whose speed counts: passes through the public entry points, as a program that serves long contexts makes them.

A case names an operation ("op"), the geometry of the model (batch, layers, query and KV heads, head_dim, dtype),
the context length N and the memory budget in per cent of the full cache:

  end_to_end        Compressor.compress, then one generated token: Compressor.append and Compressor.decode
  score             vector_score, the observation-window scorer, over the prefilled keys
  route             vector_route on given scores; with "compact" also vector_compact into the mixed cache
  route_layer       vector_route_layer: the same with one map per layer
  decode            one generation step over the mixed cache: Compressor.append and Compressor.decode
  decode_layer      the same step with one map per layer: Compressor.append and vector_decode_attn_layer

A model calls the decode step layer by layer (the next layer's queries depend on this layer's output), so one-layer
calls are as ordinary as calls that cover all layers; prefill-time compression runs either as each layer's prefill
ends or over the whole cache afterwards.
"""
import math

import torch

from paper_2605_23258_b200 import binding as B
from paper_2605_23258_b200.pipeline import Compressor

_DEVICE = "cuda"


def _case(op, batch, layers, q_heads, kv_heads, head_dim, dtype, N, window, percent, rope=False, compact=False):
    return {"op": op, "batch": batch, "layers": layers, "q_heads": q_heads, "kv_heads": kv_heads, "head_dim": head_dim,
            "dtype": dtype, "N": N, "window": window, "percent": percent, "rope": rope, "compact": compact}


def listed():
    cases = {
        # a short fp32 sequence end to end: every step of the path, all of it latency and launches
        "small_fp32_end_to_end": _case("end_to_end", 1, 1, 4, 2, 64, "fp32", 1024, 32, 25),
        # one layer scored as its prefill ends, an 8B model's attention geometry
        "score_one_layer": _case("score", 1, 1, 32, 8, 128, "bf16", 8192, 64, 20),
        # the whole prefilled cache of a 70B model's geometry at its longest context: the largest call
        "score_80_layers": _case("score", 1, 80, 64, 8, 128, "bf16", 131072, 128, 5),
        # a model with 64-channel heads, a context length that is no multiple of anything
        "score_head64_ragged": _case("score", 1, 16, 32, 8, 64, "bf16", 15013, 64, 20),
        # routing and compaction of a whole 32-layer cache
        "route_compact_32_layers": _case("route", 1, 32, 32, 8, 128, "bf16", 32768, 64, 20, compact=True),
        # routing with rotary keys, which the regressor sees turned back: four sequences, ragged length
        "route_rope_ragged": _case("route", 4, 8, 32, 8, 128, "bf16", 20011, 64, 15, rope=True),
        # routing with one map per layer
        "route_layer_map": _case("route_layer", 1, 16, 32, 8, 128, "bf16", 16384, 64, 20),
        # one layer's step of a single sequence: the latency of a generated token is this, times the layers
        "decode_one_layer": _case("decode", 1, 1, 32, 8, 128, "bf16", 8192, 64, 20),
        # batched serving, all 32 layers of eight sequences in one call
        "decode_batch8_32_layers": _case("decode", 8, 32, 32, 8, 128, "bf16", 16384, 64, 10),
        # one layer of sixteen sequences with rotary keys, ragged length
        "decode_rope_batch16": _case("decode", 16, 1, 32, 8, 128, "bf16", 30001, 64, 20, rope=True),
        # 64-channel heads, four sequences
        "decode_head64": _case("decode", 4, 16, 32, 8, 64, "bf16", 16384, 64, 20),
        # one map per layer, eight sequences, ragged length
        "decode_layer_map": _case("decode_layer", 8, 4, 32, 8, 128, "bf16", 24001, 64, 20),
    }
    return [dict(c, name=name) for name, c in cases.items()]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    """Another case of the same operations.  The number of units is cut until the pass costs no more than the largest
    listed one and the keys take at most 8 GB."""
    op = rng.choice(["end_to_end", "score", "score", "route", "route", "route_layer", "decode", "decode", "decode", "decode_layer"])
    if op == "end_to_end":
        kv_heads, g, head_dim = rng.choice([1, 2, 4]), rng.choice([1, 2, 4, 8]), rng.choice([64, 128])
        return _case(op, rng.choice([1, 2]), 1, kv_heads * g, kv_heads, head_dim, "fp32", _log_int(rng, 300, 4096), rng.choice([16, 32]), rng.choice([25, 30, 40]))
    layered = op.endswith("_layer")
    head_dim = 128 if layered else rng.choice([64, 128, 128, 128])
    kv_heads = 8 if layered else rng.choice([1, 2, 4, 8, 8])
    g = rng.choice([1, 2, 4]) if layered else rng.choice([1, 2, 3, 4, 8])
    window = rng.choice([16, 32, 48, 64, 100, 128])
    percent = rng.choice([5, 10, 15, 20, 30, 40])
    N = _log_int(rng, 2048, 65536 if layered else 131072)
    if rng.random() < 0.5:
        N = N // 128 * 128
    batch, layers = _log_int(rng, 1, 16), _log_int(rng, 1, 80)
    units_most = (8 << 30) / (2.0 * N * kv_heads * head_dim)
    if op == "score":
        units_most = min(units_most, 2e13 / (4.0 * kv_heads * g * window * N * head_dim) / (1 if head_dim == 128 else 64))
    if layered:
        units_most = min(units_most, 4e5 / N)
    while batch * layers > max(units_most, 1):
        if layers >= batch:
            layers = (layers + 1) // 2
        else:
            batch = (batch + 1) // 2
    rope = not layered and op != "score" and rng.random() < 0.5
    compact = op == "route" and head_dim == 128 and not rope
    return _case(op, batch, layers, kv_heads * g, kv_heads, head_dim, "bf16", N, window, percent, rope=rope, compact=compact)


def _shape(c):
    return B.Shape(c["batch"], c["layers"], c["q_heads"], c["kv_heads"], c["head_dim"],
                   B.VECTOR_BF16 if c["dtype"] == "bf16" else B.VECTOR_F32, c["window"], 7, 0.0, int(c["rope"]), 10000.0)


def _budget(c):
    return B.vector_plan_budget(c["N"], c["N"] * c["percent"] // 100, -1, c["window"])


class _Law:
    """The distributions of a model's cached tensors: per (layer, KV head) channel scales spread over a factor of eight,
    one key channel in a hundred twenty times larger, values a linear map of the (unrotated) key plus noise whose size
    varies from token to token, deeper layers noisier."""

    def __init__(self, c, seed):
        self.c, self.d, self.h = c, c["head_dim"], c["kv_heads"]
        self.dtype = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
        self.gen = torch.Generator(device=_DEVICE).manual_seed(seed * 7919 + 17)
        LH = c["layers"] * self.h
        self.sigma_k, self.sigma_q = self.spread((LH, self.d), 0.5, 4.0), self.spread((LH, self.d), 0.5, 4.0)
        big = torch.argsort(self.rand(LH, self.d), dim=1)[:, :max(1, self.d // 100)]
        self.sigma_k.scatter_(1, big, self.sigma_k.gather(1, big) * 20.0)

    def rand(self, *shape):
        return torch.rand(*shape, generator=self.gen, device=_DEVICE)

    def randn(self, *shape):
        return torch.randn(*shape, generator=self.gen, device=_DEVICE)

    def spread(self, shape, lo, hi):
        return torch.exp(math.log(lo) + self.rand(*shape) * math.log(hi / lo))

    def maps(self, per_layer=False):
        n, D = (self.c["layers"], self.h * self.d) if per_layer else (self.c["layers"] * self.h, self.d)
        return (self.randn(n, D, D) / math.sqrt(D)).to(self.dtype)

    def layers(self):
        """(first unit, map index of the first unit) of every (sequence, layer): the tensors are filled one at a time."""
        for bl in range(self.c["batch"] * self.c["layers"]):
            yield bl * self.h, (bl % self.c["layers"]) * self.h

    def turned(self, k, pos):
        """k [..., n, d] turned by the positions pos [..., n], channel c with c + d/2."""
        half = self.d // 2
        inv = 10000.0 ** (-2.0 * torch.arange(half, device=_DEVICE, dtype=torch.float64) / self.d)
        angle = (pos.double()[..., None] * inv).remainder(2 * math.pi).float()
        cs, sn = torch.cos(angle), torch.sin(angle)
        x, y = k[..., :half], k[..., half:]
        return torch.cat([x * cs - y * sn, x * sn + y * cs], dim=-1)

    def keys_values(self, n, W=None, pos=None, rows=None):
        """K (and V, when a map is given) [U][rows][d]; the first n rows are drawn, the rest are zero."""
        U = self.c["batch"] * self.c["layers"] * self.h
        K = torch.zeros(U, rows or n, self.d, dtype=self.dtype, device=_DEVICE)
        V = torch.zeros_like(K) if W is not None else None
        whole = W is not None and W.shape[-1] != self.d
        for u, m in self.layers():
            k = self.randn(self.h, n, self.d) * self.sigma_k[m:m + self.h, None, :]
            if W is not None:
                noise = self.spread((1 if whole else self.h, n, 1), 0.02, 2.0) * (0.05 + 1.45 * (m + 1) / (self.c["layers"] * self.h))
                if whole:
                    flat = k.to(self.dtype).permute(1, 0, 2).reshape(n, -1)
                    v = (flat @ W[m // self.h].T).float().reshape(n, self.h, self.d).permute(1, 0, 2)
                else:
                    v = torch.bmm(k.to(self.dtype), W[m:m + self.h].transpose(1, 2)).float()
                V[u:u + self.h, :n] = (v + noise * self.randn(self.h, n, self.d)).to(self.dtype)
            if self.c["rope"]:
                k = self.turned(k, pos[u:u + self.h] if pos is not None else torch.arange(n, device=_DEVICE))
            K[u:u + self.h, :n] = k.to(self.dtype)
        return K, V

    def queries(self, *per_head):
        """[U][g][...][d]"""
        g = self.c["q_heads"] // self.h
        z = self.randn(self.c["batch"], self.c["layers"] * self.h, g, *per_head, self.d)
        sigma = self.sigma_q.reshape(1, -1, *([1] * (1 + len(per_head))), self.d)
        return (z * sigma).to(self.dtype).reshape(-1, g, *per_head, self.d)

    def scores(self, units):
        """Scores as the window scorer leaves them: heavy-tailed masses, max-pooled over seven tokens, +inf in the window."""
        n = self.c["N"] - self.c["window"]
        out = torch.full((units, self.c["N"]), math.inf, device=_DEVICE)
        for u in range(0, units, 64):
            x = torch.exp(1.5 * self.randn(min(64, units - u), 1, n) - 6.0)
            out[u:u + 64, :n] = torch.nn.functional.max_pool1d(x, 7, 1, 3)[:, 0]
        return out

    def positions(self, units, n):
        """n ascending token positions below N per unit."""
        return ((torch.arange(n, device=_DEVICE) + self.rand(units, n)) * ((self.c["N"] - 1) / max(n, 1))).to(torch.int32)


def prepare(case, seed):
    law, shape, budget = _Law(case, seed), _shape(case), _budget(case)
    op, U, N, d = case["op"], shape.units, case["N"], case["head_dim"]
    s = {"op": op, "shape": shape, "budget": budget, "N": N, "compact": case["compact"]}
    if op == "score":
        s["K"], _ = law.keys_values(N)
        s["Q"] = law.queries(case["window"])
        s["scores"] = torch.empty(U, N, dtype=torch.float32, device=_DEVICE)
        s["ws"] = B.alloc_workspace(shape, budget)
        return s
    per_layer = op.endswith("_layer")
    s["W"] = law.maps(per_layer)
    if op in ("route", "route_layer", "end_to_end"):
        s["K"], s["V"] = law.keys_values(N, s["W"])
    if op in ("route", "route_layer"):
        lists = U // case["kv_heads"] if per_layer else U
        s["scores"] = law.scores(lists)
        s["tier"] = torch.empty(lists, N, dtype=torch.uint8, device=_DEVICE)
        s["ret_idx"] = torch.empty(lists, budget.n_ret, dtype=torch.int32, device=_DEVICE)
        s["apx_idx"] = torch.empty(lists, budget.n_apx, dtype=torch.int32, device=_DEVICE)
        s["eps"] = torch.empty(lists, budget.n_pool, dtype=torch.float32, device=_DEVICE)
        s["pool_idx"] = torch.empty(lists, budget.n_pool, dtype=torch.int32, device=_DEVICE)
        if case["compact"]:
            s["cache"] = B.alloc_cache(shape, budget)
        need = B.vector_workspace_bytes(shape, budget)
        if per_layer:
            need = max(need, B.vector_layer_workspace_bytes(shape, budget))
        s["ws"] = torch.empty(need, dtype=torch.uint8, device=_DEVICE)
        return s
    # generation: room for the appended rows, the step's queries and the new token's key and value
    extra = 64
    s["q"], s["out"] = law.queries(), torch.empty(U, shape.group, d, dtype=torch.bfloat16 if case["dtype"] == "bf16" else torch.float32, device=_DEVICE)
    s["k_new"], s["v_new"] = (law.randn(U, d).to(law.dtype) for _ in range(2))
    comp = s["comp"] = Compressor(shape, budget, extra_rows=extra)
    cache = comp.cache
    for t in (cache.ret_k, cache.ret_v, cache.apx_k, cache.ret_pos, cache.apx_pos):
        t.zero_()
    if op == "end_to_end":
        s["Q"] = law.queries(case["window"])
        return s
    cap = cache.ret_k.shape[1]
    ret_pos, apx_pos = law.positions(U, budget.n_ret), law.positions(U, budget.n_apx)
    cache.ret_pos[:, :budget.n_ret], cache.apx_pos[:, :budget.n_apx] = ret_pos, apx_pos
    cache.ret_k, cache.ret_v = law.keys_values(budget.n_ret, s["W"], ret_pos, cap)
    cache.apx_k = law.keys_values(budget.n_apx, None, apx_pos)[0]
    if per_layer:
        s["ws"] = torch.empty(B.vector_layer_workspace_bytes(shape, budget), dtype=torch.uint8, device=_DEVICE)
    return s


def run(s):
    op, shape, budget = s["op"], s["shape"], s["budget"]
    if op == "score":
        B.vector_score(shape, s["Q"], s["K"], s["N"], s["scores"], None, s["ws"])
        return s["scores"]
    if op in ("route", "route_layer"):
        route = B.vector_route if op == "route" else B.vector_route_layer
        route(shape, budget, s["scores"], s["K"], s["V"], s["W"], s["tier"], s["ret_idx"], s["apx_idx"], s["eps"], s["pool_idx"], s["ws"])
        # The tier map says which tokens the two index lists hold.  The lists themselves, and the rows gathered by them,
        # are returned where the residuals are sums of exact products in a fixed order: elsewhere two tokens whose
        # residuals agree to the last bits may change places, and every entry between them moves by one.
        got = {name: s[name] for name in ("tier", "eps", "pool_idx")}
        if s["compact"]:
            c = s["cache"]
            B.vector_compact(shape, budget, s["K"], s["V"], s["ret_idx"], s["apx_idx"], c)
            got.update(ret_idx=s["ret_idx"], apx_idx=s["apx_idx"], ret_k=c.ret_k, ret_v=c.ret_v, apx_k=c.apx_k, ret_pos=c.ret_pos, apx_pos=c.apx_pos)
        return got
    comp = s["comp"]
    cache = comp.cache
    got = {}
    if op == "end_to_end":
        comp.compress(s["Q"], s["K"], s["V"], s["W"])
        got = {"scores": comp.scores, "tier": comp.tier, "ret_idx": comp.ret_idx, "apx_idx": comp.apx_idx, "apx_k": cache.apx_k, "apx_pos": cache.apx_pos}
    else:
        cache.n_ret = budget.n_ret              # every pass is the first token after the prefill
    comp.append(s["k_new"], s["v_new"], s["N"])
    if op == "decode_layer":
        B.vector_decode_attn_layer(shape, s["q"], cache, s["W"], s["out"], s["ws"])
    else:
        comp.decode(s["q"], s["W"], s["out"])
    got.update(out=s["out"], ret_k=cache.ret_k, ret_v=cache.ret_v, ret_pos=cache.ret_pos)
    return got


def work(case):
    """Each input read once, each output written once; the products the method itself asks for."""
    shape, b = _shape(case), _budget(case)
    U, N, d, g, w = shape.units, case["N"], case["head_dim"], shape.group, case["window"]
    es = 2 if case["dtype"] == "bf16" else 4
    lists = U // case["kv_heads"] if case["op"].endswith("_layer") else U
    D = case["kv_heads"] * d if case["op"].endswith("_layer") else d
    maps = case["layers"] * (D * D if case["op"].endswith("_layer") else case["kv_heads"] * d * d) * es
    row = d * es
    score = {"bytes": U * (N * row + g * w * row + 4 * N), "flops": 2.0 * U * g * w * N * d}
    route = {"bytes": lists * (4 * N + N + 4 * (b.n_ret + b.n_apx) + 8 * b.n_pool) + U * 2 * b.n_pool * row + maps,
             "flops": 2.0 * lists * b.n_pool * D * D}
    compact = {"bytes": U * (2 * (2 * b.n_ret + b.n_apx) * row + 4 * (b.n_ret + b.n_apx)), "flops": 0.0}
    decode = {"bytes": U * ((2 * b.n_ret + b.n_apx) * row + 6 * row + 2 * g * row) + maps,
              "flops": U * g * (4.0 * (b.n_ret + 1) * d + 2.0 * b.n_apx * (d + D) + 2.0 * D * d)}
    parts = {"score": [score], "route": [route], "route_layer": [route], "decode": [decode], "decode_layer": [decode],
             "end_to_end": [score, route, compact, decode]}[case["op"]]
    if case["compact"]:
        parts = parts + [compact]
    return {"bytes": float(sum(p["bytes"] for p in parts)), "flops": float(sum(p["flops"] for p in parts))}


def tolerance(case):
    """Measured against the same formulas in fp64 on the listed cases' inputs (relative 2-norm): scores 9e-7 (3e-6 at
    most for one score), residuals 1e-6 per head and 3e-6 with one map per layer, 8e-5 with keys turned back (the turned
    key is kept to 2^-17), attention 1.9e-3 (the rounding of a bf16 output), 2e-7 in fp32.  A tier changes where two
    tokens' residuals lie closer than that to the cut."""
    op = case["op"]
    if op in ("score", "end_to_end"):
        return {"rel": 5e-6}
    if op == "route" and case["rope"]:
        return {"rel": 3e-4, "differ": 1e-4}
    if op in ("route", "route_layer"):
        return {"rel": 1e-5, "differ": 2e-5}
    return {"rel": 4e-3}
