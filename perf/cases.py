"""What a user of this package has it do, as cases that can be timed and compared.

Three paths, each through the package's public calls:

  compact   after a prompt has been prefilled: per layer the last token's query scores the eviction region, the best
            tokens are selected and the reduced cache is gathered (SageKV.score, optionally SageKV's pooled scores,
            SageKV.select_compact).  Needed once per prompt and layer, and again at every refresh.
  decode    generating tokens: per layer and token one append to the recent window and one attention over the reduced
            cache (SageKV.decode_attn), called one by one or replayed from a CUDA graph of the whole stack.
  quest     one decode step of the block-wise comparator: bounds of all blocks, then the best blocks per query head.

A case is a dict of plain values:
  path, layers, q_heads, kv_heads, batch, n_ctx (tokens, the last one included), budget (rows of the reduced cache
  without the last token), split ("fixed": 4 sink tokens and 128 recent ones; "paper": a quarter of the budget each),
  and the options of the path: hint, phases, pooled (compact); graph, overlap, lse (decode).
"""

import math

import torch

from paper_2503_08879_b200 import binding as B
from paper_2503_08879_b200 import synth

LLAMA = dict(q_heads=32, kv_heads=8)      # Llama-3.1-8B, Llama-3-8B
QWEN = dict(q_heads=28, kv_heads=4)       # Qwen2.5-7B: seven query heads per KV head

DEV = "cuda"


def _compact(name, shape, n_ctx, budget, layers=1, batch=1, split="fixed", hint=0, phases=False, pooled=False):
    c = dict(path="compact", layers=layers, batch=batch, n_ctx=n_ctx, budget=budget, split=split, hint=hint, phases=phases,
             pooled=pooled, **shape)
    return dict(c, name=name) if name else c


def _decode(name, shape, budget, layers=1, batch=1, split="fixed", graph=False, overlap=0, lse=False):
    # the prompt only has to be long enough to select from: what decode touches is the reduced cache
    c = dict(path="decode", layers=layers, batch=batch, n_ctx=2 * budget, budget=budget, split=split, graph=graph,
             overlap=overlap, lse=lse, **shape)
    return dict(c, name=name) if name else c


def _quest(name, shape, n_ctx, budget, layers=1, batch=1):
    c = dict(path="quest", layers=layers, batch=batch, n_ctx=n_ctx, budget=budget, split="fixed", **shape)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one short prompt, one layer, every option at its default: all launch latency and host work
        _compact("compact-4k", LLAMA, 4096, 512),
        # a medium prompt with the paper's own split of the budget, an odd length, a batch of two, four layers
        _compact("compact-29k-b2-paper", LLAMA, 29333, 8192, layers=4, batch=2, split="paper"),
        # the long-document prompt the package is quoted on, layer by layer with the default options
        _compact("compact-128k", LLAMA, 131072, 2048, layers=2),
        # the same with everything the package offers: scores of all layers first, then all selections from the lists
        _compact("compact-128k-list", LLAMA, 131072, 2048, layers=4, hint=2, phases=True),
        # the longest prompts and the largest budget, with the histogram hint
        _compact("compact-512k-hist", LLAMA, 524288, 8192, hint=1),
        # seven query heads per KV head, a batch of four prompts of odd length, one selection per KV head
        _compact("compact-qwen-100k-b4-pooled", QWEN, 100003, 2048, batch=4, pooled=True),
        # one decode call on a small reduced cache, defaults, straight from Python
        _decode("decode-512", LLAMA, 512),
        # a token through a whole stack at batch 1, replayed from a graph: the usual serving loop
        _decode("decode-2048-stack", LLAMA, 2048, layers=32, graph=True, overlap=2),
        # the same with the largest budget
        _decode("decode-8192-stack", LLAMA, 8192, layers=32, graph=True, overlap=2),
        # a small batch on the seven-heads-per-KV-head shape
        _decode("decode-qwen-2048-b4-stack", QWEN, 2048, layers=28, batch=4, graph=True, overlap=2),
        # a serving batch, called from Python with default options, log-sum-exps wanted as well
        _decode("decode-2048-b32", LLAMA, 2048, layers=4, batch=32, lse=True),
        # one step of the comparator over a long prompt
        _quest("quest-128k", LLAMA, 131072, 2048, layers=2),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    shape = rng.choice([LLAMA, LLAMA, QWEN, dict(q_heads=16, kv_heads=2), dict(q_heads=16, kv_heads=8)])
    kind = rng.choice(["compact"] * 4 + ["decode"] * 5 + ["quest"])
    split = rng.choice(["fixed", "paper"])
    if kind == "compact":
        n_ctx = _log_int(rng, 2048, 524288)
        budget = _log_int(rng, 256, min(8192, n_ctx // 2))
        tokens = 524288 * 8 // (n_ctx * shape["kv_heads"])       # K rows of a pass against the largest listed case
        batch = min(tokens, rng.choice([1, 1, 2, 3, 4]))
        layers = max(1, min(4, tokens // batch))
        hint = rng.choice([0, 0, 1, 2])
        return _compact(None, shape, n_ctx, budget, layers, batch, split, hint, phases=hint == 2 or rng.random() < 0.3,
                        pooled=hint == 0 and rng.random() < 0.2)
    if kind == "decode":
        budget = _log_int(rng, 256, 8192)
        batch = _log_int(rng, 1, 48)
        layers = max(1, min(32, 32 * 8192 * 8 // (budget * batch * shape["kv_heads"])))
        layers = rng.randint(1, layers)
        graph = rng.random() < 0.6
        overlap = rng.choice([0, 1, 2]) if layers > 1 else rng.choice([0, 1])
        return _decode(None, shape, budget, layers, batch, split, graph, overlap, lse=rng.random() < 0.3)
    n_ctx = _log_int(rng, 16384, 262144)
    return _quest(None, shape, n_ctx, _log_int(rng, 512, 8192), layers=rng.randint(1, 2), batch=rng.randint(1, 2))


def _workload(case, seed):
    """The case as a workload of the package's input generator: random keys with planted heavy tokens."""
    G = case["q_heads"] // case["kv_heads"]
    n_init, n_recent = 4, 128
    if case["split"] == "paper":
        n_init, _, n_recent = B.sagekv_budget_split(case["budget"], G)
    return synth.Workload("case", case["layers"], case["q_heads"], case["kv_heads"], 128, case["batch"], case["n_ctx"],
                          case["budget"], n_init, n_recent, 1, "varfrac", (0.001, 0.02), seed=int(seed))


def _context(case, w):
    return B.SageKV(w.n_q_heads, w.n_kv_heads, w.head_dim, w.batch, max_ctx=w.n_ctx, max_len=w.L, device=DEV)


def _prepare_compact(case, seed):
    w = _workload(case, seed)
    sk = _context(case, w)
    sk.set_select_hint(case["hint"], w.n_sel)
    if case["pooled"]:
        B.sagekv_set_group_mode(sk.ctx, 1)
    if case["phases"] and w.n_layers > 1:
        sk.set_select_overlap(2)        # the kernel before a select call is another layer's, or another layer's score call
    st = dict(case=case, w=w, sk=sk, layers=[])
    for l in range(w.n_layers):
        lay = synth.make_layer(w, l, DEV)
        lay.pop("heavy")
        lay["scores"] = sk.new_scores(w.n_ctx, w.n_init, w.n_recent)
        if case["pooled"]:
            lay["pooled"] = torch.empty(w.batch * w.n_kv_heads, lay["scores"].stride(0), device=DEV)
            lay["cache"] = B.Layer(w.batch, w.n_kv_heads, w.n_kv_heads, w.head_dim, w.L, w.n_sel, DEV)
        else:
            lay["cache"] = sk.new_layer(w.n_init, w.n_recent, w.n_sel)
        st["layers"].append(lay)
    return st


def _run_compact(st):
    w, sk, case = st["w"], st["sk"], st["case"]

    def score(lay):
        sk.score(lay["q_last"], lay["K"], w.n_init, w.n_recent, lay["scores"])

    def select(lay):
        rows = lay["scores"]
        if case["pooled"]:
            B.sagekv_pool_scores(sk.ctx, rows, rows.stride(0), w.n_ctx, w.n_init, w.n_recent, lay["pooled"],
                                 lay["pooled"].stride(0))
            rows = lay["pooled"]
        sk.select_compact(rows, lay["K"], lay["V"], w.n_init, w.n_recent, w.n_sel, lay["cache"])

    if case["phases"]:
        for lay in st["layers"]:
            score(lay)
        for lay in st["layers"]:
            select(lay)
    else:
        for lay in st["layers"]:
            score(lay)
            select(lay)
    return [(lay["scores"][:, : w.E], lay["cache"].idx, lay["cache"].Kc, lay["cache"].Vc) for lay in st["layers"]]


def _prepare_decode(case, seed):
    w = _workload(case, seed)
    sk = _context(case, w)
    sk.set_overlap(case["overlap"])
    n, Bt, Hq, Hkv, d = w.n_layers, w.batch, w.n_q_heads, w.n_kv_heads, w.head_dim
    bf16 = dict(dtype=torch.bfloat16, device=DEV)
    # the serving program keeps the caches and the activations of all layers in one tensor each
    st = dict(case=case, w=w, sk=sk, caches=[], Kc=torch.empty(n, Bt, Hkv, w.L, d, **bf16),
              Vc=torch.empty(n, Bt, Hkv, w.L, d, **bf16), q=torch.empty(n, Bt, Hq, d, **bf16),
              k_new=torch.empty(n, Bt, Hkv, d, **bf16), v_new=torch.empty(n, Bt, Hkv, d, **bf16),
              out=torch.empty(n, Bt, Hq, d, **bf16), lse=torch.empty(n, Bt, Hq, device=DEV) if case["lse"] else None)
    scores = sk.new_scores(w.n_ctx, w.n_init, w.n_recent)
    for l in range(n):
        lay = synth.make_layer(w, l, DEV)
        cache = sk.new_layer(w.n_init, w.n_recent, w.n_sel)
        cache.Kc, cache.Vc = st["Kc"][l], st["Vc"][l]
        sk.score(lay["q_last"], lay["K"], w.n_init, w.n_recent, scores)
        sk.select_compact(scores, lay["K"], lay["V"], w.n_init, w.n_recent, w.n_sel, cache)
        st["caches"].append(cache)
        for name, x in synth.make_decode_inputs(w, l, 0, DEV).items():
            st[name][l].copy_(x)
    if case["graph"]:
        saved = [x.clone() for x in (st["Kc"], st["Vc"])]
        _decode_stack(st)               # once outside the capture: loads the kernels
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            _decode_stack(st)
        st["graph"] = graph
        for x, y in zip((st["Kc"], st["Vc"]), saved):
            x.copy_(y)
        for cache in st["caches"]:
            cache.step.zero_()
    return st


def _decode_stack(st):
    lse = st["lse"]
    for l, cache in enumerate(st["caches"]):
        st["sk"].decode_attn(st["q"][l], st["k_new"][l], st["v_new"][l], cache, st["out"][l], None if lse is None else lse[l])


def _run_decode(st):
    if st["case"]["graph"]:
        st["graph"].replay()
    else:
        _decode_stack(st)
    return [st[k] for k in ("out", "lse", "Kc", "Vc") if st[k] is not None]


def _prepare_quest(case, seed):
    w = _workload(case, seed)
    n_blocks = (w.E + 15) // 16
    sk = _context(case, w)
    st = dict(case=case, w=w, sk=sk, n_blocks=n_blocks, k=min(n_blocks, max(1, w.k_q // 16)), layers=[])
    for l in range(w.n_layers):
        lay = synth.make_layer(w, l, DEV)
        s = dict(q=synth.make_decode_inputs(w, l, 0, DEV)["q"])
        s["kmin"] = torch.empty(w.batch, w.n_kv_heads, n_blocks, w.head_dim, dtype=torch.bfloat16, device=DEV)
        s["kmax"] = torch.empty_like(s["kmin"])
        B.sagekv_quest_build(sk.ctx, lay["K"], w.n_ctx, w.n_init, w.n_recent, s["kmin"], s["kmax"])
        s["bounds"] = torch.empty(w.batch * w.n_q_heads, (n_blocks + 3) // 4 * 4, device=DEV)
        s["idx"] = torch.empty(w.batch, w.n_q_heads, st["k"], dtype=torch.int32, device=DEV)
        st["layers"].append(s)
    return st


def _run_quest(st):
    sk, n = st["sk"], st["n_blocks"]
    for s in st["layers"]:
        B.sagekv_quest_bounds(sk.ctx, s["q"], s["kmin"], s["kmax"], n, s["bounds"], s["bounds"].stride(0))
        B.sagekv_select_topk(sk.ctx, s["bounds"], s["bounds"].stride(0), n, st["k"], s["idx"])
    return [(s["bounds"][:, :n], s["idx"]) for s in st["layers"]]


def prepare(case, seed):
    with torch.cuda.device(DEV):
        return {"compact": _prepare_compact, "decode": _prepare_decode, "quest": _prepare_quest}[case["path"]](case, seed)


def run(state):
    return {"compact": _run_compact, "decode": _run_decode, "quest": _run_quest}[state["case"]["path"]](state)


def work(case):
    w = _workload(case, 0)
    row = w.head_dim * 2                                              # bytes of one key or value
    n = w.n_layers * w.batch
    if case["path"] == "compact":
        heads = w.n_kv_heads if case["pooled"] else w.n_q_heads
        kept = w.n_kv_heads * w.L * row                               # of K, and of V
        read = w.n_kv_heads * (w.E + w.n_init + w.n_recent + 1) * row + kept + w.n_q_heads * row
        written = w.n_q_heads * w.E * 4 + 2 * kept + heads * (w.n_sel * w.n_kv_heads // heads) * 4
        return {"bytes": n * (read + written), "flops": n * 2 * w.n_q_heads * w.E * w.head_dim}
    if case["path"] == "decode":
        seen = w.n_init + w.k_q + w.n_recent + 1                      # rows one query head attends to
        small = 2 * w.n_q_heads * row + 4 * w.n_kv_heads * row + (4 * w.n_q_heads if case["lse"] else 0)
        return {"bytes": n * (2 * w.n_kv_heads * w.L * row + small), "flops": n * 4 * w.n_q_heads * seen * w.head_dim}
    blocks = (w.E + 15) // 16
    k = min(blocks, max(1, w.k_q // 16))
    return {"bytes": n * (w.n_kv_heads * blocks * 2 * row + w.n_q_heads * (row + blocks * 4 + k * 4)),
            "flops": n * 4 * w.n_q_heads * blocks * w.head_dim}


def tolerance(case):
    if case["path"] == "decode":
        # bf16 outputs and bf16 softmax weights, each half an ulp (2^-9 of a value) off at most; measured against
        # 64-bit attention over the same caches: 2.2e-3, largest 1.5e-2
        return {"rel": 9e-3, "max": 6e-2}
    # fp32 sums of 128 bf16 products, exp2 to about 2 ulp; measured against 64-bit softmax rows: 3.4e-7, largest
    # 1.4e-6 (block bounds: 4.7e-8, 1.7e-7).  A whole value differs where two scores tie within that.
    return {"rel": 1.5e-6, "max": 6e-6, "differ": 1e-2}
