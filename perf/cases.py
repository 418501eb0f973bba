"""What a program has the library do, as cases to time and to compare.

A case is one kind of call at one shape:

  decode   one token through every layer with the inputs on the GPU
  host     the same from and to page-locked host memory
  full     the same with every token kept (no eviction)
  realloc  an adaptive budget reallocation and the tokens up to the next one
  prompt   a new batch: its handle, the prompts of all layers, the first token, and the handle freed
  window   the same with an observation window

The calls go through the C ABI of the loaded library with addresses as a serving loop holds them.
Prompts are N(0, 1) rows with an attention sink (key 0 times 8) and outlier keys (times 3, 0.5 to 5
per cent of a head's keys).  The rows that arrive step by step are windows of a bank of such rows
that move by one row per layer and step, so that no head meets the same key twice.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2601_16986_b200 import EVICT, FULLKV, Config, CrystalKV

D = 128
BANK = 1 << 16          # distinct positions of the arriving rows
PROMPTS = 4             # distinct layers' prompts that a new batch takes in turn
CONTEXT = 1 << 18       # longest trajectory of a handle that is stepped on and on (its size does not depend on it)
THINK = 1 << 14         # think tokens that a handle made for a new batch of prompts is sized for
FULL_ROOM = 2048        # tokens a full cache may grow by while it is in use
TOP_P = 0.9


def _case(name, kind, layers, q_heads, kv_heads, batch, budget, prompt, unequal=False, every=0, window=0, ratio=0.0,
          evict_every=1):
    c = {"kind": kind, "layers": layers, "q_heads": q_heads, "kv_heads": kv_heads, "batch": batch, "budget": budget,
         "prompt": prompt, "unequal": unequal, "every": every, "window": window, "ratio": ratio, "evict_every": evict_every}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one layer, one sequence; latency of the launch chain and of the call itself
        _case("decode_1layer_batch1", "decode", 1, 8, 2, 1, 512, 512),
        # the 7B shape at its usual batch: 32 heads per launch, few bytes
        _case("decode_7b_batch8", "decode", 28, 28, 4, 8, 1024, 1024),
        # the 8B shape with budgets as reallocations leave them: heads of very different lengths
        _case("decode_8b_batch16_unequal", "decode", 32, 32, 8, 16, 2048, 0, unequal=True),
        # the 14B shape with such budgets: the default workload of the benchmark
        _case("decode_14b_batch32_unequal", "decode", 48, 40, 8, 32, 1024, 0, unequal=True),
        # few sequences with a large budget
        _case("decode_14b_batch8_budget4096", "decode", 48, 40, 8, 8, 4096, 4096),
        # many sequences with a small budget: about as many heads as warps
        _case("decode_14b_batch128_budget256", "decode", 48, 40, 8, 128, 256, 256),
        # the full-cache baseline at the 8K reasoning level
        _case("full_8b_batch16_9350", "full", 32, 32, 8, 16, 1024, 9350),
        # a program that keeps its activations on the host
        _case("host_7b_batch8", "host", 28, 28, 4, 8, 1024, 1024),
        # budgets that are adapted often
        _case("realloc_14b_batch8_every16", "realloc", 48, 40, 8, 8, 1024, 1024, every=16),
        # a prompt that fits the budget
        _case("prompt_8b_batch16_512", "prompt", 32, 32, 8, 16, 2048, 512),
        # a long prompt under the 10 per cent ratio rule: scored, cut to 935 entries per head
        _case("prompt_8b_batch8_9350_ratio", "prompt", 32, 32, 8, 8, 1024, 9350, ratio=0.1),
        # a prompt scored by its last 32 queries
        _case("window_14b_batch16_1024_w32", "window", 48, 40, 8, 16, 1024, 1024, window=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["decode", "host", "full", "realloc", "prompt", "window"], [10, 2, 2, 2, 4, 2])[0]
    while True:
        kv = rng.choice([1, 2, 4, 8])
        g = rng.randint(1, 8)
        layers, batch = _log(rng, 1, 48), _log(rng, 1, 128)
        budget = _log(rng, 100, 4096)
        heads = layers * batch * kv
        if batch * kv > 1024 or heads * budget * 512 > 7e9:
            continue
        if kind in ("decode", "host"):
            unequal = rng.random() < 0.5
            return _case(None, kind, layers, g * kv, kv, batch, budget, 0 if unequal else budget, unequal=unequal,
                         evict_every=rng.choice([1, 1, 1, 16]))
        if kind == "full":
            prompt = _log(rng, 300, 20000)
            if heads * (prompt + FULL_ROOM) * 512 < 20e9 and heads * prompt * 512 > 2e9:
                return _case(None, kind, layers, g * kv, kv, batch, budget, prompt)
        if kind == "realloc":
            every = rng.randint(8, 64)
            if every * heads * budget * 512 < 20e9:
                return _case(None, kind, layers, g * kv, kv, batch, budget, budget, every=every)
        if kind == "prompt":
            prompt = _log(rng, 100, 12000)
            ratio = rng.choice([0.0, 0.1, 0.25])
            if batch * kv * prompt * 512 < 4e8 and prompt < 4 * budget:
                return _case(None, kind, layers, g * kv, kv, batch, budget, prompt, ratio=ratio)
        if kind == "window":
            window = _log(rng, 1, 64)
            if layers * window * batch * kv * budget * 512 < 2e11 and layers * window * batch * kv * g < 4e5:
                prompt = rng.randint(max(64, budget // 2), budget)
                return _case(None, kind, layers, g * kv, kv, batch, budget, prompt, window=window)


# ---------------------------------------------------------------- inputs
def _gen(seed, salt, device="cuda"):
    return torch.Generator(device).manual_seed((seed * 1000003 + salt) & 0x7FFFFFFFFFFFFFFF)


def _rows(shape, g):
    return torch.randn(*shape, D, dtype=torch.bfloat16, device="cuda", generator=g)


def _budgets(case, seed):
    """Budgets [batch, layers, kv_heads] as reallocations leave them: half to one and a half times the mean."""
    shape = (case["batch"], case["layers"], case["kv_heads"])
    if not case["unequal"]:
        return np.full(shape, case["budget"], dtype=np.int64)
    f = np.random.RandomState((seed * 7919 + 17) & 0x7FFFFFFF).uniform(0.5, 1.5, shape)
    return np.maximum(1, np.floor(case["budget"] * f / f.mean(axis=(1, 2), keepdims=True))).astype(np.int64)


def _prompt_len(case, budgets):
    return case["prompt"] or int(budgets.max())


def _prompt(case, seed, layer, P):
    """k, v [batch, P, kv_heads, 128] and the last prompt queries [max(window, 1), batch, q_heads, 128]."""
    g = _gen(seed, 100 + layer)
    shape = (case["batch"], P, case["kv_heads"])
    k, v = _rows(shape, g), _rows(shape, g)
    frac = 0.005 + 0.045 * torch.rand(case["kv_heads"], device="cuda", generator=g)
    scale = torch.where(torch.rand(shape, device="cuda", generator=g) < frac, 3.0, 1.0)
    scale[:, 0] = 8.0
    k.mul_(scale.unsqueeze(-1).to(torch.bfloat16))
    return k, v, _rows((max(case["window"], 1), case["batch"], case["q_heads"]), g)


def _bank(case, seed):
    """The rows that arrive: queries, keys, values; the call at step i of layer l takes consecutive rows from (i L + l) mod BANK."""
    g = _gen(seed, 1)
    q = _rows((BANK + case["batch"] * case["q_heads"],), g)
    k = _rows((BANK + case["batch"] * case["kv_heads"],), g)
    v = _rows((BANK + case["batch"] * case["kv_heads"],), g)
    k.mul_(torch.where(torch.rand(k.shape[0], 1, device="cuda", generator=g) < 0.03, 3.0, 1.0).to(torch.bfloat16))
    return q, k, v


# ---------------------------------------------------------------- state
class _State:
    pass


def _ok(s, rc):
    if rc:
        raise RuntimeError(s.kv.lib.crystalkv_last_error(s.kv._h).decode())


def _handle(case, P):
    full = case["kind"] == "full"
    context = {"full": P + FULL_ROOM, "prompt": P + THINK, "window": P + THINK}.get(case["kind"], CONTEXT)
    return CrystalKV(Config(n_layers=case["layers"], n_q_heads=case["q_heads"], n_kv_heads=case["kv_heads"],
                            batch=case["batch"], budget_per_head=case["budget"],
                            max_context=context, mode=FULLKV if full else EVICT,
                            top_p=TOP_P, max_budget=max(4 * case["budget"], P), evict_every=case["evict_every"],
                            budget_ratio=case["ratio"]))


def prepare(case, seed):
    s = _State()
    s.case, s.kind = case, case["kind"]
    L, B, Hq, H = case["layers"], case["batch"], case["q_heads"], case["kv_heads"]
    budgets = _budgets(case, seed)
    s.P = P = _prompt_len(case, budgets)
    s.bank = _bank(case, seed)
    s.stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    s.step = 0
    if s.kind in ("prompt", "window"):
        s.prompts = [_prompt(case, seed, i, P) for i in range(min(L, PROMPTS))]
        s.out = torch.empty(1, L, B, Hq, D, dtype=torch.bfloat16, device="cuda")
        s.out_window = torch.empty(L, case["window"], B, Hq, D, dtype=torch.bfloat16, device="cuda")
    else:
        s.kv = _handle(case, P)
        for l in range(L):
            if case["unequal"]:
                for b in range(B):
                    for h in range(H):
                        s.kv.set_budget(l, b, h, int(budgets[b, l, h]))
            k, v, q = _prompt(case, seed, l, P)
            s.kv.prefill(l, k, v, q[0])
        tokens = max(case["every"], 1)
        s.out = torch.empty(tokens, L, B, Hq, D, dtype=torch.bfloat16, device="cuda")
        if s.kind == "host":
            s.bank = tuple(x.cpu().pin_memory() for x in s.bank)
            s.out = torch.empty(tokens, L, B, Hq, D, dtype=torch.bfloat16).pin_memory()
    s.addr = [x.data_ptr() for x in s.bank]
    s.out_addr, s.out_bytes = s.out.data_ptr(), B * Hq * D * 2
    torch.cuda.synchronize()
    return s


def _token(s, i):
    """One token through every layer; its outputs go to s.out[i]."""
    kv, st, L = s.kv, s.stream, s.case["layers"]
    call = kv.lib.crystalkv_decode_step_host if s.kind == "host" else kv.lib.crystalkv_decode_step
    h, (q, k, v) = kv._h, s.addr
    out = s.out_addr + i * L * s.out_bytes
    at = s.step * L
    for l in range(L):
        o = ((at + l) % BANK) * 256
        _ok(s, call(h, l, q + o, k + o, v + o, out, st))
        out += s.out_bytes
    s.step += 1


def _new_batch(s):
    """A new batch of prompts: a handle of its own, every layer's prompt, the first token."""
    c = s.case
    s.kv, s.step = _handle(c, s.P), 0
    lib, h = s.kv.lib, s.kv._h
    for l in range(c["layers"]):
        k, v, q = (x.data_ptr() for x in s.prompts[l % len(s.prompts)])
        if s.kind == "window":
            _ok(s, lib.crystalkv_prefill_window(h, l, k, v, q, s.P, c["window"], s.out_window[l].data_ptr(), s.stream))
        else:
            _ok(s, lib.crystalkv_prefill(h, l, k, v, q, s.P, s.stream))
    _token(s, 0)
    s.kv.close()


def run(s):
    if s.kind in ("prompt", "window"):
        _new_batch(s)
        return {"out": s.out, "window": s.out_window} if s.kind == "window" else s.out
    if s.kind == "realloc":
        _ok(s, s.kv.lib.crystalkv_rebudget(s.kv._h, s.stream))
    for i in range(max(s.case["every"], 1)):
        _token(s, i)
    if s.kind == "host":   # the results are read on the host
        _ok(s, s.kv.lib.crystalkv_join(s.kv._h, s.stream))
        torch.cuda.current_stream().synchronize()
    return s.out


# ---------------------------------------------------------------- what a pass needs
def _kept(case):
    """Entries per head, on average, that a token finds."""
    P = case["prompt"]
    if case["kind"] == "full":
        return P
    if case["kind"] == "prompt":
        return min(P, _ratio_budget(case) if case["ratio"] else case["budget"])
    return case["budget"] if not P else min(P, case["budget"])


def _ratio_budget(case):
    b = math.floor(float(np.float32(case["ratio"])) * case["prompt"])
    low = min(case["budget"], max(16, case["budget"] // 8))
    return min(max(b, low), case["budget"])


def work(case):
    """K and V rows, CRF and last hit time (read) of every entry; queries, outputs and arriving rows; two products of G x 128."""
    U, Hq, P, n = case["batch"] * case["kv_heads"], case["batch"] * case["q_heads"], case["prompt"], _kept(case) + 1
    meta = 0 if case["kind"] == "full" else 8
    token = {"bytes": U * n * (512 + meta) + Hq * 512 + U * 1024, "flops": Hq * n * 4 * D}
    if case["kind"] in ("prompt", "window"):
        w = max(case["window"], 1)
        # every key is read, the survivors' values are read, the survivors are stored
        return {"bytes": case["layers"] * (U * (P * 256 + n * 256 + n * 524) + w * Hq * 512 + token["bytes"]),
                "flops": case["layers"] * (w * Hq * P * (4 if case["window"] else 2) * D + token["flops"])}
    m = case["layers"] * max(case["every"], 1)
    again = case["layers"] * U * n * 8 if case["kind"] == "realloc" else 0   # the aggregation of CRF
    return {"bytes": m * token["bytes"] + again, "flops": m * token["flops"]}


def tolerance(case):
    # outputs are rounded to bf16 (relative 2-norm 1.7e-3 against 64 bits); one entry more or fewer at the
    # hit boundary of a head moves that head's outputs by the weight of one entry
    return {"rel": 7e-3, "max": 0.1}


# ---------------------------------------------------------------- the same in 64 bits
def _attend(q, k, v, live=None):
    """q [w, b, Hq, D], k and v [b, n, H, D], live [w or 1, b, H, n] or None -> probabilities, outputs [w, b, Hq, D]."""
    w, b, Hq, _ = q.shape
    H = k.shape[2]
    x = torch.einsum("wbhgd,bnhd->wbhgn", q.double().view(w, b, H, Hq // H, D), k.double()) / math.sqrt(D)
    if live is not None:
        x = x.masked_fill(~live.unsqueeze(3), -math.inf)
    p = torch.softmax(x, -1)
    return p, torch.einsum("wbhgn,bnhd->wbhgd", p, v.double()).reshape(w, b, Hq, D)


def _survivors(k, v, q, budget):
    """bool [b, H, P]: what is left of a prompt once its last query has marked hits (the smallest set of the likeliest
    entries that reaches the threshold) and the lowest, misses first and then the earliest, have left; budget [b, H]."""
    p = _attend(q, k, v)[0][0].mean(2)
    val, order = p.sort(dim=-1, descending=True, stable=True)
    before = val.cumsum(-1) - val
    hit = torch.zeros_like(p, dtype=torch.bool).scatter_(-1, order, before < float(np.float32(TOP_P)) * val.sum(-1, keepdim=True))
    P = p.shape[-1]
    key = hit.long() * P + torch.arange(P, device="cuda")
    least = key.sort(-1, descending=True)[0].gather(-1, (budget.clamp(max=P) - 1).unsqueeze(-1))
    return key >= least


def exact(case, seed):
    if case["kind"] == "realloc":
        return None
    budgets = _budgets(case, seed)
    P, kind = _prompt_len(case, budgets), case["kind"]
    L, B, Hq, H = case["layers"], case["batch"], case["q_heads"], case["kv_heads"]
    qb, kb, vb = _bank(case, seed)
    got, seen = [], []
    for l in range(L):
        k, v, q = _prompt(case, seed, l % PROMPTS if kind in ("prompt", "window") else l, P)
        if kind == "window":
            t = torch.arange(P, device="cuda")
            live = t <= (P - case["window"] + torch.arange(case["window"], device="cuda")).unsqueeze(1)
            if l < PROMPTS:
                seen.append(torch.cat([_attend(q[i:i + 1], k, v, live[i].view(1, 1, 1, P))[1] for i in range(len(q))]))
            continue
        b = torch.from_numpy(budgets[:, l]).cuda()
        if kind == "prompt" and case["ratio"]:
            b = torch.full_like(b, _ratio_budget(case))
        if kind == "full":
            b = torch.full_like(b, P)
        live = _survivors(k, v, q, b) if P > int(b.min()) else torch.ones(B, H, P, dtype=torch.bool, device="cuda")
        live = live | (P - b < case["evict_every"]).unsqueeze(-1)   # not yet over by a whole period: nothing has left
        live = torch.cat([live, torch.ones_like(live[..., :1])], -1).unsqueeze(0)
        q1 = qb[l:l + B * Hq].view(1, B, Hq, D)
        k1, v1 = (x[l:l + B * H].view(B, 1, H, D) for x in (kb, vb))
        got.append(_attend(q1, torch.cat([k, k1], 1), torch.cat([v, v1], 1), live)[1][0])
    if kind == "window":
        return {"out": None, "window": torch.stack([seen[l % PROMPTS].float() for l in range(L)])}
    return torch.stack(got).unsqueeze(0)
