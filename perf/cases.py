"""The work that is timed: what a program that generates step by step has this library do, through its public calls.

Every case is a dict of plain values; `op` names the path:

  token        one decode token over the layers of a model (Context.decode_step / _e4m3 / _i4, one call per layer)
  host_token   the same token's attention with the per-step tensors in host memory (attn_host_begin / attn_host_wait)
  step         a batch of steps scored and routed: cache write, chunk attention, router head, rollback of the rejected
               (kv_append, attn, route, rollback); with no prefix and no head it is the prefill of prompts
  draft_step   what a draft's cache sees of an escalated step: tokens one by one, rollback, the target's step as a chunk
  serving      one iteration of a serving loop: decode rows and step chunks of one batch in one attention call
  loop         one round of Algorithm 1 over draft, router and target caches (step_loop.StepLoop)
  router_eval  escalation policies and Spearman's rho over the steps of an evaluation split

Lengths are spread evenly over a case's range (a lognormal one by its quantiles), so that the work of a case does not
depend on the seed; the seed gives the order of the sequences, the pages and every value.
"""
import math
import random
import statistics

import torch

from paper_2512_05033_b200 import binding
from paper_2512_05033_b200.step_loop import Cache, StepLoop

PAGE = 16
BF16, F32 = torch.bfloat16, torch.float32
GEOMETRIES = ((12, 2), (28, 4), (32, 8))   # query / KV heads: draft-, router- and target-shaped
SCALE = 0.0125                             # of an E4M3 cache: N(0, 1) rows use the middle of the code range
TAU = 0.5

_ctx = None


def _context():
    global _ctx
    if _ctx is None:
        _ctx = binding.Context(0)
    return _ctx


# ---- the cases ----------------------------------------------------------------------------------------------------

def _token(name, kv, B, heads, lo, hi, layers, head_dim=128):
    return {"name": name, "op": "token", "kv": kv, "batch": B, "hq": heads[0], "hkv": heads[1], "head_dim": head_dim,
            "lo": lo, "hi": hi, "layers": layers}


def _host_token(name, B, heads, lo, hi, layers):
    return {"name": name, "op": "host_token", "kv": "bf16", "batch": B, "hq": heads[0], "hkv": heads[1], "head_dim": 128,
            "lo": lo, "hi": hi, "layers": layers}


def _step(name, kv, B, heads, lo, hi, n_lo, n_hi, hidden, head_dim=128):
    return {"name": name, "op": "step", "kv": kv, "batch": B, "hq": heads[0], "hkv": heads[1], "head_dim": head_dim,
            "lo": lo, "hi": hi, "n_lo": n_lo, "n_hi": n_hi, "hidden": hidden}


def _draft_step(name, kv, B, heads, lo, hi, tokens, n_lo, n_hi, head_dim=128):
    return {"name": name, "op": "draft_step", "kv": kv, "batch": B, "hq": heads[0], "hkv": heads[1],
            "head_dim": head_dim, "lo": lo, "hi": hi, "tokens": tokens, "n_lo": n_lo, "n_hi": n_hi}


def _serving(name, B, heads, lo, hi, n_lo, n_hi):
    return {"name": name, "op": "serving", "kv": "bf16", "batch": B, "hq": heads[0], "hkv": heads[1], "head_dim": 128,
            "lo": lo, "hi": hi, "n_lo": n_lo, "n_hi": n_hi, "hidden": 3584}


def _loop(name, kv, B, lo, hi, n_lo, n_hi):
    return {"name": name, "op": "loop", "kv": kv, "batch": B, "lo": lo, "hi": hi, "n_lo": n_lo, "n_hi": n_hi,
            "hidden": 3584}


def _router_eval(name, n):
    return {"name": name, "op": "router_eval", "n": n}


def listed():
    return [
        # the smallest call: one sequence, fp32, a 16-token step scored and routed (the configuration parity is pinned on)
        _step("tiny_step", "fp32", 1, (8, 2), 512, 512, 16, 16, 256, head_dim=64),
        # a draft token: the latency of this call times tokens times layers is the draft's share of the loop
        _token("draft_token", "bf16", 8, (12, 2), 1024, 8192, 28),
        # a target token over long contexts: as many bytes as a decode call of this loop moves
        _token("target_token", "bf16", 16, (32, 8), 4096, 32768, 2),
        # a draft token over the 4-bit cache
        _token("i4_token", "i4", 8, (12, 2), 1024, 8192, 28),
        # a draft token of a program whose per-step tensors live in host memory
        _host_token("host_token", 8, (12, 2), 1024, 8192, 28),
        # the router's forward over a batch of finished steps, its decision, and the rollback
        _step("step_scoring", "bf16", 32, (28, 4), 2048, 16384, 16, 128, 3584),
        # a quantised draft: tokens over the E4M3 cache, then the target's step absorbed as a chunk
        _draft_step("e4m3_draft_step", "e4m3", 16, (12, 2), 2048, 8192, 16, 8, 32),
        # a small draft model with 64-dimension heads doing the same
        _draft_step("head64_draft_step", "bf16", 16, (32, 8), 1024, 8192, 16, 8, 32, head_dim=64),
        # continuous batching: half the batch decodes, half scores a step, lengths lognormal
        _serving("mixed_serving", 64, (32, 8), 256, 65536, 16, 128),
        # a whole round of Algorithm 1
        _loop("step_loop", "bf16", 16, 2048, 8192, 8, 32),
        # the prompts of a batch enter a cache
        _step("prefill", "bf16", 8, (32, 8), 0, 0, 256, 2048, 0),
        # a router judged on an evaluation split: every policy with its statistics, and the rank correlation
        _router_eval("router_eval", 20000),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        case = _draw(rng)
        case.pop("name")
        if _cost(case) <= most and _cache_bytes(case) <= 6e9:
            return case


def _draw(rng):
    op = rng.choice(("token", "token", "token", "host_token", "step", "step", "step", "draft_step", "draft_step",
                     "serving", "loop", "prefill", "router_eval"))
    heads = rng.choice(GEOMETRIES)
    hi = _log_int(rng, 256, 32768)
    lo = max(16, hi // rng.choice((1, 4, 8)))
    if op == "token":
        kv = rng.choice(("bf16", "bf16", "e4m3", "i4"))
        return _token("", kv, _log_int(rng, 1, 32), heads, lo, hi, rng.choice((2, 7, 16, 28)),
                      head_dim=64 if kv == "bf16" and rng.random() < 0.25 else 128)
    if op == "host_token":
        return _host_token("", _log_int(rng, 1, 16), heads, max(16, lo // 4), hi // 4, rng.choice((16, 28)))
    if op == "step":
        kv = rng.choice(("bf16", "bf16", "bf16", "e4m3", "fp32"))
        n_hi = _log_int(rng, 8, 128)
        n_lo = max(2, n_hi // 4)
        if kv == "fp32":
            return _step("", kv, rng.randint(1, 2), (8, 2), max(16, lo // 16), max(16, hi // 16), n_lo, n_hi, 256,
                         head_dim=rng.choice((64, 128)))
        return _step("", kv, _log_int(rng, 1, 48), heads, lo, hi, n_lo, n_hi, 3584,
                     head_dim=64 if kv == "bf16" and rng.random() < 0.25 else 128)
    if op == "draft_step":
        kv = rng.choice(("bf16", "bf16", "e4m3", "e4m3"))
        n_hi = _log_int(rng, 8, 64)
        return _draft_step("", kv, _log_int(rng, 1, 24), heads, max(16, lo // 2), hi // 2, _log_int(rng, 4, 32),
                           max(2, n_hi // 4), n_hi, head_dim=64 if kv == "bf16" and rng.random() < 0.5 else 128)
    if op == "serving":
        return _serving("", _log_int(rng, 4, 64), heads, 256, 65536, 16, _log_int(rng, 32, 128))
    if op == "loop":
        n_hi = _log_int(rng, 8, 32)
        return _loop("", rng.choice(("bf16", "e4m3")), _log_int(rng, 1, 24), max(16, lo // 4), max(256, hi // 4),
                     max(2, n_hi // 4), n_hi)
    if op == "prefill":
        n_hi = _log_int(rng, 128, 4096)
        return _step("", rng.choice(("bf16", "bf16", "e4m3")), _log_int(rng, 1, 16), heads, 0, 0, max(2, n_hi // 8), n_hi, 0)
    return _router_eval("", _log_int(rng, 256, 40000))


# ---- lengths and work ---------------------------------------------------------------------------------------------

def _spread(count, lo, hi):
    """`count` whole numbers spread evenly over lo .. hi."""
    return [lo + int((hi - lo) * (i + 0.5) / count) for i in range(count)]


def _prefixes(case):
    B = case["batch"]
    if case["op"] == "serving":   # lognormal, median 8192, sigma 0.8 in log space
        z = [statistics.NormalDist().inv_cdf((i + 0.5) / B) for i in range(B)]
        return [max(case["lo"], min(case["hi"], int(round(8192 * math.exp(0.8 * v))))) for v in z]
    return _spread(B, case["lo"], case["hi"])


def _steps(case, salt=0):
    """Step lengths, in an order of their own."""
    B = case["batch"]
    n = _spread(B, case["n_lo"], case["n_hi"])
    random.Random(1000 * B + salt).shuffle(n)
    if case["op"] == "serving":
        n = [1 if i % 2 == 0 else v for i, v in enumerate(n)]
    return n


def _kv_bytes_per_token(case, heads=None, kv=None):
    """Bytes of keys and values of one token in one layer's cache."""
    hkv, d = (case["hkv"], case["head_dim"]) if heads is None else (heads[1], 128)
    per_row = {"fp32": 4 * d, "bf16": 2 * d, "e4m3": d, "i4": d // 2 + 4}[kv or case["kv"]]
    return 2 * hkv * per_row


def _attn_work(prefixes, steps, hq, hkv, d, esz, kv_tok, written=True):
    """Bytes and flops of one attention call with the cache write in front of it."""
    n, kv = sum(steps), sum(p + s for p, s in zip(prefixes, steps))
    pairs = sum(s * p + s * (s + 1) // 2 for p, s in zip(prefixes, steps))
    pages = sum((p + s + PAGE - 1) // PAGE for p, s in zip(prefixes, steps))
    b = kv * kv_tok + 2 * n * hq * d * esz + 4 * pages + 8 * len(steps)
    if written:   # the new rows are read once more from k_new / v_new
        b += 2 * n * hkv * d * esz
    return b, 4 * pairs * hq * d


def work(case):
    op = case["op"]
    if op == "router_eval":
        n = case["n"]   # two scores in, five decision vectors and the statistics out; the sorts
        return {"bytes": 8 * n + 4 * n + 8 * n, "flops": 4 * 10 * n * math.log2(n)}
    prefixes = _prefixes(case)
    if op == "loop":
        return _loop_work(case, prefixes)
    hq, hkv, d = case["hq"], case["hkv"], case["head_dim"]
    esz = 4 if case["kv"] == "fp32" else 2
    kv_tok = _kv_bytes_per_token(case)
    one = [1] * len(prefixes)
    if op in ("token", "host_token"):
        b, f = _attn_work(prefixes, one, hq, hkv, d, esz, kv_tok, op == "token")
        return {"bytes": b * case["layers"], "flops": f * case["layers"]}
    b, f = _attn_work(prefixes, _steps(case), hq, hkv, d, esz, kv_tok)
    if op == "draft_step":
        for t in range(case["tokens"]):
            bt, ft = _attn_work([p + t for p in prefixes], one, hq, hkv, d, esz, kv_tok)
            b, f = b + bt, f + ft
    elif case["hidden"]:
        b += case["batch"] * case["hidden"] * esz
        f += 2 * case["batch"] * case["hidden"]
    return {"bytes": b, "flops": f}


def _loop_work(case, prefixes):
    """Half of the steps escalate (hidden . w is symmetric around the threshold)."""
    sd, st = _steps(case), _steps(case, 7)
    draft, router, target = GEOMETRIES
    kv = [_kv_bytes_per_token(case, g, k) for g, k in zip(GEOMETRIES, (case["kv"], "bf16", "bf16"))]
    b = f = 0.0

    def tokens(steps, g, kv_tok, share):
        nonlocal b, f
        for p, s in zip(prefixes, steps):
            for t in range(s):
                bt, ft = _attn_work([p + t], [1], g[0], g[1], 128, 2, kv_tok)
                b, f = b + share * bt, f + share * ft

    def chunk(steps, g, kv_tok, share):
        nonlocal b, f
        bc, fc = _attn_work(prefixes, steps, g[0], g[1], 128, 2, kv_tok)
        b, f = b + share * bc, f + share * fc

    tokens(sd, draft, kv[0], 1.0)
    chunk(sd, router, kv[1], 1.0)
    chunk(sd, target, kv[2], 0.5)
    tokens(st, target, kv[2], 0.5)
    chunk(st, router, kv[1], 0.5)
    chunk(st, draft, kv[0], 0.5)
    b += case["batch"] * case["hidden"] * 2
    return {"bytes": b, "flops": f}


def _cost(case):
    w = work(case)
    # fp32 and 64-dimension chunks and the policies' comparisons run on the CUDA cores: their operations weigh more
    slow = case["op"] == "router_eval" or case["kv"] == "fp32" or case.get("head_dim") == 64
    return max(w["bytes"], w["flops"] / (5 if slow else 200))


def _cache_bytes(case):
    if case["op"] == "router_eval":
        return 0
    tokens = sum(_prefixes(case)) + 160 * case["batch"]
    if case["op"] == "loop":
        return tokens * sum(_kv_bytes_per_token(case, g, "bf16") for g in GEOMETRIES)
    return tokens * _kv_bytes_per_token(case) * case.get("layers", 1)


def tolerance(case):
    if case["op"] == "router_eval":   # decisions and counters are whole numbers; the sums are 64-bit, in any order
        return {"rel": 1e-10}
    if case["kv"] == "fp32":          # 32-bit sums: 2.2e-7 (largest 9e-7) against 64 bits on tiny_step, more on longer rows
        return {"rel": 3e-6, "max": 3e-5}
    # bf16 rows out and softmax weights of 8 bits (11 over codes): 1.7e-3 to 2.4e-3 (largest element 0.028) against 64 bits
    # on the same cache; cache contents, lengths and decisions are exact
    return {"rel": 1e-2, "max": 0.1}


# ---- inputs -------------------------------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _normal(gen, shape, dtype=BF16):
    return torch.randn(shape, generator=gen, device="cuda", dtype=dtype)


def _ints(values):
    return torch.tensor(values, dtype=torch.int32, device="cuda")


def _pages(lens, rng):
    """A block table over a shuffled pool with room for `lens` tokens per sequence, and the pool's pages."""
    need = [(n + PAGE - 1) // PAGE for n in lens]
    total = sum(need) + 3
    order = list(range(total))
    rng.shuffle(order)
    table = torch.full((len(lens), max(need)), -1, dtype=torch.int32)
    at = 0
    for b, n in enumerate(need):
        table[b, :n] = torch.tensor(order[at:at + n], dtype=torch.int32)
        at += n
    return table.cuda(), total


def _pools(kv, layers, pages, hkv, d, gen):
    """K and V pools of `layers` layers, filled as a cache in use is (and, for a 4-bit cache, their scale pools)."""
    shape = (layers, pages, hkv, PAGE, d)
    if kv == "e4m3":
        return [(_normal(gen, shape) / SCALE).to(torch.float8_e4m3fn).view(torch.uint8) for _ in range(2)]
    if kv == "i4":
        half = shape[:-1] + (d // 2,)
        codes = []
        for _ in range(2):
            lo, hi = ((_normal(gen, half) * 2.5).round_().clamp_(-7, 7).to(torch.int32) + 8 for _ in range(2))
            codes.append((lo | (hi << 4)).to(torch.uint8))
        scales = [torch.rand(shape[:-1], generator=gen, device="cuda") * 0.1 + 0.35 for _ in range(2)]
        return codes + scales
    return [_normal(gen, shape, F32 if kv == "fp32" else BF16) for _ in range(2)]


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case, s.ctx = case, _context()
    gen, rng = _gen(seed), random.Random(seed)
    return {"token": _prepare_token, "host_token": _prepare_host_token, "step": _prepare_step,
            "draft_step": _prepare_draft_step, "serving": _prepare_step, "loop": _prepare_loop,
            "router_eval": _prepare_router_eval}[case["op"]](s, case, gen, rng)


def _shuffled(rng, *lists):
    order = list(range(len(lists[0])))
    rng.shuffle(order)
    return [[v[i] for i in order] for v in lists]


def _prepare_token(s, case, gen, rng):
    B, L, hq, hkv, d = (case[k] for k in ("batch", "layers", "hq", "hkv", "head_dim"))
    prefixes, = _shuffled(rng, _prefixes(case))
    s.table, pages = _pages([p + 1 for p in prefixes], rng)
    s.pools = _pools(case["kv"], L, pages, hkv, d, gen)
    q = _normal(gen, (L, B, hq, d))
    k, v = _normal(gen, (L, B, hkv, d)), _normal(gen, (L, B, hkv, d))
    s.out = torch.zeros_like(q)
    s.start = _ints([prefixes] * L)
    s.lens = s.start.clone()
    s.ones = _ints([1] * B)
    s.layers = [(q[i], k[i], v[i], *(p[i] for p in s.pools), s.lens[i], s.out[i]) for i in range(L)]
    return s


def _prepare_host_token(s, case, gen, rng):
    B, L, hq, hkv, d = (case[k] for k in ("batch", "layers", "hq", "hkv", "head_dim"))
    prefixes, = _shuffled(rng, _prefixes(case))
    table, pages = _pages([p + 1 for p in prefixes], rng)
    s.pools = _pools("bf16", L, pages, hkv, d, gen)
    q = _normal(gen, (L, B, hq, d)).cpu().pin_memory()
    s.out = torch.zeros_like(q).pin_memory()
    s.table = table.cpu().pin_memory()
    s.lens = torch.tensor([p + 1 for p in prefixes], dtype=torch.int32).pin_memory()
    s.ones = torch.ones(B, dtype=torch.int32).pin_memory()
    s.layers = [(q[i], s.pools[0][i], s.pools[1][i], s.out[i]) for i in range(L)]
    return s


def _prepare_step(s, case, gen, rng):
    B, hq, hkv, d = (case[k] for k in ("batch", "hq", "hkv", "head_dim"))
    dt = F32 if case["kv"] == "fp32" else BF16
    prefixes, steps = _shuffled(rng, _prefixes(case), _steps(case))
    s.table, pages = _pages([p + n for p, n in zip(prefixes, steps)], rng)
    s.k, s.v = (p[0] for p in _pools(case["kv"], 1, pages, hkv, d, gen))
    n = sum(steps)
    s.q = _normal(gen, (n, hq, d), dt)
    s.k_new, s.v_new = _normal(gen, (n, hkv, d), dt), _normal(gen, (n, hkv, d), dt)
    s.out = torch.zeros_like(s.q)
    s.start, s.steps, s.most = _ints(prefixes), _ints(steps), max(steps)
    s.lens = s.start.clone()
    if case["hidden"]:
        _router(s, case, gen, dt)
        s.scored = _ints([n if n > 1 else 0 for n in steps])   # a sequence that decodes has no step to roll back
    return s


def _router(s, case, gen, dt):
    B, H = case["batch"], case["hidden"]
    s.hidden = _normal(gen, (B, H), dt)
    s.w = (_normal(gen, (H,), F32) / math.sqrt(H)).to(dt)
    s.scores = torch.zeros(B, dtype=F32, device="cuda")
    s.decisions = torch.zeros(B, dtype=torch.uint8, device="cuda")


def _prepare_draft_step(s, case, gen, rng):
    B, T, hq, hkv, d = (case[k] for k in ("batch", "tokens", "hq", "hkv", "head_dim"))
    prefixes, steps = _shuffled(rng, _prefixes(case), _steps(case))
    s.table, pages = _pages([p + max(n, T) for p, n in zip(prefixes, steps)], rng)
    s.k, s.v = (p[0] for p in _pools(case["kv"], 1, pages, hkv, d, gen))
    q, k, v = _normal(gen, (T, B, hq, d)), _normal(gen, (T, B, hkv, d)), _normal(gen, (T, B, hkv, d))
    s.token_out = torch.zeros_like(q)
    s.tokens = [(q[t], k[t], v[t], s.token_out[t]) for t in range(T)]
    n = sum(steps)
    s.q = _normal(gen, (n, hq, d))
    s.k_new, s.v_new = _normal(gen, (n, hkv, d)), _normal(gen, (n, hkv, d))
    s.out = torch.zeros_like(s.q)
    s.start, s.steps, s.most = _ints(prefixes), _ints(steps), max(steps)
    s.lens = s.start.clone()
    s.ones, s.written = _ints([1] * B), _ints([T] * B)
    return s


def _prepare_loop(s, case, gen, rng):
    B, d = case["batch"], 128
    most = case["n_hi"]
    prefixes, step_d, step_t = _shuffled(rng, _prefixes(case), _steps(case), _steps(case, 7))
    s.caches, s.start = [], _ints(prefixes)
    for (hq, hkv), kv in zip(GEOMETRIES, (case["kv"], "bf16", "bf16")):
        table, pages = _pages([p + 2 * most for p in prefixes], rng)
        k, v = (p[0] for p in _pools(kv, 1, pages, hkv, d, gen))
        s.caches.append(Cache(hq, k, v, table, s.start.clone(), e4m3=(SCALE, SCALE) if kv == "e4m3" else None))
    _router(s, case, gen, BF16)
    s.step_d, s.step_t = _ints(step_d), _ints(step_t)
    s.loop = StepLoop(s.ctx, *s.caches, s.w, 0.0, TAU, max(step_d), max(step_t))

    def rows(n, g, per_token):
        shape = (n, B) if per_token else (n * B,)
        return tuple(_normal(gen, shape + (h, d)) for h in (g[0], g[1], g[1]))

    draft, router, target = GEOMETRIES
    nd, nt = s.loop.nd, s.loop.nt
    s.acts = {"draft.gen": rows(nd, draft, True), "target.gen": rows(nt, target, True),
              "router.zd": rows(nd, router, False), "target.zd": rows(nd, target, False),
              "router.zt": rows(nt, router, False), "draft.zt": rows(nt, draft, False)}
    s.outs = {}
    for name, (q, _, _) in s.acts.items():   # one buffer per phase
        s.outs[name] = torch.zeros_like(q)
        if name.endswith(".gen"):
            s.loop.out.update({f"{name}[{t}]": s.outs[name][t] for t in range(q.shape[0])})
        else:
            s.loop.out[name] = s.outs[name]
    return s


def _prepare_router_eval(s, case, gen, rng):
    n = case["n"]
    skill = _normal(gen, (n,), F32)   # PRM scores: correlated, in (0, 1), kept to four digits as scores are
    s.s_d = (torch.sigmoid(skill + 0.7 * _normal(gen, (n,), F32)) * 1e4).round_() / 1e4
    s.s_t = (torch.sigmoid(skill + 0.4 + 0.7 * _normal(gen, (n,), F32)) * 1e4).round_() / 1e4
    s.advantage = s.s_t - s.s_d
    s.router = torch.sigmoid(0.3 * s.advantage + 0.5 * _normal(gen, (n,), F32))
    s.kinds = [(binding.POLICY_RSD, 0.5, 0), (binding.POLICY_ORACLE_THRESHOLD, 0.1, 0),
               (binding.POLICY_ORACLE_ARGMAX, 0.0, 0), (binding.POLICY_ORACLE_BUDGET, 0.0, n // 4)]
    s.decisions = torch.zeros(len(s.kinds), n, dtype=torch.uint8, device="cuda")
    s.stats = torch.zeros(len(s.kinds), 3, dtype=torch.float64, device="cuda")
    s.rho = torch.zeros(1, dtype=torch.float64, device="cuda")
    return s


# ---- one pass -----------------------------------------------------------------------------------------------------

def run(s):
    return {"token": _run_token, "host_token": _run_host_token, "step": _run_step, "draft_step": _run_draft_step,
            "serving": _run_step, "loop": _run_loop, "router_eval": _run_router_eval}[s.case["op"]](s)


def _decode(s, q, k_new, v_new, pools, lens, out):
    kv = s.case["kv"]
    if kv == "e4m3":
        s.ctx.decode_step_e4m3(q, k_new, v_new, *pools, SCALE, SCALE, 1.0 / SCALE, 1.0 / SCALE, s.table, lens, s.ones, out=out)
    elif kv == "i4":
        s.ctx.decode_step_i4(q, k_new, v_new, *pools, s.table, lens, s.ones, out=out)
    else:
        s.ctx.decode_step(q, k_new, v_new, *pools, s.table, lens, s.ones, out=out)


def _absorb(s):
    """The cache takes the new rows of every sequence, and the step's queries attend."""
    if s.case["kv"] == "e4m3":
        s.ctx.kv_append_e4m3(s.k_new, s.v_new, 1.0 / SCALE, 1.0 / SCALE, s.table, s.lens, s.steps, s.k, s.v)
        s.ctx.attn_e4m3(s.q, s.k, s.v, SCALE, SCALE, s.table, s.lens, s.steps, s.most, out=s.out)
    else:
        s.ctx.kv_append(s.k_new, s.v_new, s.table, s.lens, s.steps, s.k, s.v)
        s.ctx.attn(s.q, s.k, s.v, s.table, s.lens, s.steps, s.most, out=s.out)


def _run_token(s):
    s.lens.copy_(s.start)   # every pass generates the same token
    for q, k_new, v_new, *pools, lens, out in s.layers:
        _decode(s, q, k_new, v_new, pools, lens, out)
    return {"out": s.out, "lens": s.lens, "pools": s.pools}


def _run_host_token(s):
    for q, k, v, out in s.layers:
        s.ctx.attn_host_begin(q, k, v, s.table, s.lens, s.ones, 1, out, flags=binding.ATTN_OVERLAP_PREVIOUS)
    s.ctx.attn_host_wait()
    return s.out


def _run_step(s):
    s.lens.copy_(s.start)
    _absorb(s)
    got = {"out": s.out, "k": s.k, "v": s.v, "lens": s.lens}
    if s.case["hidden"]:
        s.ctx.route(s.hidden, s.w, 0.0, TAU, scores=s.scores, decisions=s.decisions)
        s.ctx.rollback(s.lens, s.scored, s.decisions)
        got.update(scores=s.scores, decisions=s.decisions)
    return got


def _run_draft_step(s):
    s.lens.copy_(s.start)
    for q, k_new, v_new, out in s.tokens:
        _decode(s, q, k_new, v_new, (s.k, s.v), s.lens, out)
    s.ctx.rollback(s.lens, s.written)   # the step was escalated: the draft forgets it ...
    _absorb(s)                          # ... and takes the target's
    return {"tokens": s.token_out, "out": s.out, "k": s.k, "v": s.v, "lens": s.lens}


def _run_loop(s):
    for c in s.caches:
        c.seq_lens.copy_(s.start)
    decisions = s.loop.round(s.step_d, s.step_t, s.hidden, s.acts)
    return {"decisions": decisions, "scores": s.loop.scores, "outs": s.outs,
            "caches": [(c.k_pages, c.v_pages, c.seq_lens) for c in s.caches]}


def _run_router_eval(s):
    for i, (kind, tau, budget) in enumerate(s.kinds):
        s.ctx.policy(kind, s.s_d, s.s_t, tau, budget, decisions=s.decisions[i], stats=s.stats[i])
    s.ctx.spearman(s.router, s.advantage, rho=s.rho)
    return {"decisions": s.decisions, "counts": s.stats[:, :1].contiguous().view(torch.int32), "sums": s.stats[:, 1:], "rho": s.rho}
